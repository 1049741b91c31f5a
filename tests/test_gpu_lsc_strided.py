"""Gradients of a layer whose input's rows are further apart than its own voxels need (a range of
voxels of a larger activation): the same as those of a compact copy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("start,V", [(0, 200), (136, 77)])
def test_lsc_backward_of_a_voxel_range(dtype, start, V):
    dirs, bvals = synth.multishell_table([40, 40], [1000, 2000], seed=41)
    lb = L.SHBasis(dirs, bvals, 8, 0.006)
    lg = L.LSCGeometry(lb, 4, 2, np.deg2rad(25), 2, 6, "same")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")  # noqa: E731
    ci, co = 3, 5
    x = layers.as_act(rnd(2 * ci * lg.n_in, 512).to(dtype))[:, start:start + V]
    assert x.stride(0) == 512
    w, d = rnd(co, 2, ci, 2, lg.K), layers.as_act(rnd(2 * co * lg.n_out, V).to(dtype))
    got = layers.lsc_backward(lg, x, w, d, ci, co)
    want = layers.lsc_backward(lg, x.clone(memory_format=torch.contiguous_format), w, d, ci, co)
    L.check_device_error("strided input")
    assert all(torch.equal(a, b) for a, b in zip(got, want))
