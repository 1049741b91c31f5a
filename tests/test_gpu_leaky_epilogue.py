"""The leaky ReLU and its adjoint in the LSC GEMMs' epilogues: bit for bit the two passes they
replace (the value is rounded to the activation type first, as a pass would read it), over the
staged and direct epilogues, ragged tiles and the paths that run a pass after all; and the
network's stack of layers against its modules called one by one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402
from paper_1808_01517_gb300 import net as N  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    # staged forward; direct input gradient through W, and from 8,192 voxels on through its transpose
    "16_to_24": dict(m=[40, 40, 40], ci=16, co=24, order_in=8, s_in=3, win="adjacent", V=1000),
    "16_to_24_transposed": dict(m=[40, 40, 40], ci=16, co=24, order_in=8, s_in=3, win="adjacent", V=8203),
    # staged input gradient (K = 90 .. 135), a ragged last tile with a partial 16-byte chunk
    "64_to_1": dict(m=[40, 40, 40], ci=64, co=1, order_in=8, s_in=3, win="adjacent", V=777),
    # one input shell, padded operator rows
    "1_to_20": dict(m=[40, 40, 40], ci=1, co=20, order_in=4, s_in=1, win="all", V=515),
    # padded shell blocks: the forward reads Wt
    "5_to_7": dict(m=[40, 40], ci=5, co=7, order_in=6, s_in=2, win="same", V=130),
}


@pytest.mark.parametrize("mode,cluster", [(L.TC_PREFER, 2), (L.TC_PREFER, 1), (L.TC_OFF, 2)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("case", list(CASES))
def test_epilogue_equals_the_passes(case, dtype, mode, cluster, gemm_cluster):
    c = CASES[case]
    gemm_cluster(cluster)
    S = len(c["m"])
    dirs, bvals = synth.multishell_table(c["m"], [1000, 2000, 3000][:S], seed=41)
    lb = L.SHBasis(dirs, bvals, 8, 0.006)
    lg = L.LSCGeometry(lb, c["order_in"], c["s_in"], np.deg2rad(25), 2, 6, c["win"])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    x = layers.as_act(rnd(c["s_in"] * c["ci"] * lg.n_in, c["V"]).to(dtype))
    x[::7, ::3] = 0.0  # zeros take the slope
    w, b = rnd(c["co"], S, c["ci"], c["s_in"], lg.K), rnd(c["co"], S)
    d = layers.as_act(rnd(S * c["co"] * lg.n_out, c["V"]).to(dtype))
    L.set_tensor_cores(mode)
    try:
        y = layers.leaky_relu(layers.lsc_forward(lg, x, w, b, c["ci"], c["co"]), 0.1)
        y2 = layers.lsc_forward(lg, x, w, b, c["ci"], c["co"], slope=0.1)
        dx, dw, db = layers.lsc_backward(lg, x, w, d, c["ci"], c["co"])
        dx2, dw2, db2 = layers.lsc_backward(lg, x, w, d, c["ci"], c["co"], slope=0.1)
    finally:
        L.set_tensor_cores(True)
    L.check_device_error(case)
    want = torch.where(x.float() > 0, dx.float(), (0.1 * dx.float()).to(dtype).float()).to(dtype)
    assert torch.equal(y, y2)
    assert torch.equal(want, dx2)
    assert torch.equal(dw, dw2) and torch.equal(db, db2)


def test_stack_equals_its_modules():
    cfg = N.NetConfig(hidden=8, dirs_per_shell=(40, 40, 40), rings=2, sectors=6)
    dirs, bvals, sel = N.tables(cfg)
    m = N.SphericalNet(cfg, dirs[sel], dirs, bvals).cuda()
    x = torch.rand((len(sel), 333), device="cuda").bfloat16()

    def grads(pred):
        return torch.autograd.grad(pred.float().square().sum(), list(m.parameters()))

    pred = m(x)
    got = grads(pred)
    seen = []
    handle = m.act.register_forward_hook(lambda *a: seen.append(1))  # a hook: the modules are called
    ref = m(x)
    want = grads(ref)
    assert len(seen) == cfg.n_lsc - 1
    handle.remove()
    assert torch.equal(pred, ref) and all(torch.equal(a, b) for a, b in zip(got, want))
    with torch.no_grad():
        assert torch.equal(m(x), ref)
