"""FP32 layer backward in a buffer without the room for the transposed operator parts at its end (the
size the call needed before it made them): taken, with the same gradients; anything less is refused.

Tolerance of the relative L2 difference of the input gradients: the same six part products over
tiles of another width, each within about 1e-6 of FP64: 2e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,extra", [(4096, True), (4099, True), (4095, False)])
def test_backward_without_the_transposed_parts(V, extra):
    ci, co = 16, 8
    dirs, bvals = synth.multishell_table([60], [1000], seed=3)
    lb = L.SHBasis(dirs, bvals, 8, 0.006)
    lg = L.LSCGeometry(lb, 8, 1, np.deg2rad(25), 2, 6, "same")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    x, d = layers.as_act(rnd(ci * lg.n_in, V)), layers.as_act(rnd(co * lg.n_out, V))
    w = rnd(co, 1, ci, 1, lg.K) / 30
    keep, ptr, full = layers.lsc_workspace(lg, V, ci, co, torch.float32, True)
    parts = -(-6 * ci * lg.n_in * co * lg.n_out // 256) * 256 if extra else 0
    want = layers.lsc_backward(lg, x, w, d, ci, co, workspace=(keep, ptr, full))
    got = layers.lsc_backward(lg, x, w, d, ci, co, workspace=(keep, ptr, full - parts))
    L.check_device_error("backward")
    for a, b in zip(got, want):
        assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) <= 2e-6
    with pytest.raises(L.DelimitError) as e:
        layers.lsc_backward(lg, x, w, d, ci, co, workspace=(keep, ptr, full - parts - 1))
    assert e.value.status == L.ERR_WORKSPACE
