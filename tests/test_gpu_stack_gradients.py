"""Gradients of the network's stack of layers, where hooks on the parameters or a process group may
follow them, arrive layer by layer, last layer first, each before the backward of the layer below
it runs (what overlaps a gradient exchange with the backward); frozen layers are left out; and both
forms of the stack give the same bits."""
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import layers  # noqa: E402
from paper_1808_01517_gb300 import net as N  # noqa: E402

pytestmark = pytest.mark.gpu


def _net():
    cfg = N.NetConfig(hidden=8, dirs_per_shell=(40, 40, 40), rings=2, sectors=6)
    dirs, bvals, sel = N.tables(cfg)
    m = N.SphericalNet(cfg, dirs[sel], dirs, bvals).cuda()
    return m, torch.rand((len(sel), 333), device="cuda").bfloat16()


def _events(monkeypatch, m):
    events, run = [], layers.lsc_backward
    index = {id(lsc.geom): i for i, lsc in enumerate(m.lscs)}

    def logged(geom, *args, **kw):
        events.append(("backward", index[id(geom)]))
        return run(geom, *args, **kw)

    monkeypatch.setattr(layers, "lsc_backward", logged)
    for i, lsc in enumerate(m.lscs):
        for p in (lsc.weight, lsc.bias):
            if p.requires_grad:
                p.register_post_accumulate_grad_hook(lambda p, i=i: events.append(("grad", i)))
    return events


def test_gradients_arrive_with_their_layer(monkeypatch):
    m, x = _net()
    events = _events(monkeypatch, m)
    m(x).float().square().sum().backward()
    want = []
    for i in reversed(range(len(m.lscs))):
        want += [("backward", i), ("grad", i), ("grad", i)]
    assert events == want


@pytest.mark.parametrize("frozen", [(0, 1), (1, 3), (3,)])
def test_frozen_layers(monkeypatch, frozen):
    m, x = _net()
    for i in frozen:
        m.lscs[i].requires_grad_(False)
    params = [p for p in m.parameters() if p.requires_grad]
    handle = m.act.register_forward_hook(lambda *a: None)  # a hook: the modules are called one by one
    want = torch.autograd.grad(m(x).float().square().sum(), params)
    handle.remove()
    got = torch.autograd.grad(m(x).float().square().sum(), params)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    first = min(i for i in range(len(m.lscs)) if i not in frozen)
    events = _events(monkeypatch, m)
    m(x).float().square().sum().backward()
    assert [i for k, i in events if k == "backward"] == list(reversed(range(first, len(m.lscs))))


def test_a_process_group_is_someone_who_follows(tmp_path):
    """Data-parallel wrappers hook the gradients where the parameters do not show it."""
    dist = torch.distributed
    m, x = _net()

    def nodes(y):
        names, todo, seen = [], [y.grad_fn], set()
        while todo:
            f = todo.pop()
            if f is not None and f not in seen:
                seen.add(f)
                names.append(type(f).__name__)
                todo += [n for n, _ in f.next_functions]
        return names.count("_LSCFnBackward"), names.count("_LSCStackFnBackward")

    alone = m(x)
    assert nodes(alone) == (0, 1)
    want = torch.autograd.grad(alone.float().square().sum(), list(m.parameters()))
    dist.init_process_group("gloo", init_method=f"file://{tmp_path}/store", rank=0, world_size=1)
    try:
        y = m(x)
    finally:
        dist.destroy_process_group()
    assert nodes(y) == (len(m.lscs), 0)
    got = torch.autograd.grad(y.float().square().sum(), list(m.parameters()))
    assert torch.equal(y, alone) and all(torch.equal(a, b) for a, b in zip(got, want))
