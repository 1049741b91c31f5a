"""The weight gradient's reduction on the tensor cores where a voxel sum is infinite, undefined or
larger than the largest BF16 value (it is split into BF16 parts there): infinities keep their sign,
NaN stays NaN, large finite sums stay finite, and nothing spreads to other channel pairs.  The CUDA
cores' FP32 sum of the same inputs is the reference; finite values agree to the tolerance of
test_gpu_reduce_dw_route.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu

BIG = 181 / 128 * 2.0 ** 63  # twice its square, 1.9996 2^127, lies between the largest BF16 and FP32 values
# the voxel sum of one pair of rows as the product (dY, X) of one voxel
SUMS = {
    "inf": (1e25, 1e25),
    "-inf": (1e25, -1e25),
    "nan": (float("nan"), 1.0),
    "large": (BIG, 2 * BIG),
    "-large": (-BIG, 2 * BIG),
}


@pytest.mark.parametrize("order", [4, 8, 10])  # one, three and five k-steps per input coefficient
@pytest.mark.parametrize("kind", list(SUMS))
def test_as_the_fp32_sum(kind, order):
    ci, co, V, m = 3, 20, 16, [70, 70]
    dirs, bvals = synth.multishell_table(m, [1000, 2000], seed=33)
    lb = L.SHBasis(dirs, bvals, order, 0.006)
    lg = L.LSCGeometry(lb, order, 2, np.deg2rad(25), 2, 6, "all")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x = torch.randn((2 * ci * lg.n_in, V), generator=gen, device="cuda").bfloat16()
    d = torch.randn((2 * co * lg.n_out, V), generator=gen, device="cuda").bfloat16()
    r, c = (co + 11) * lg.n_out + lg.n_out // 2, lg.n_in + 3  # shell 1 of channel 11, shell 0 of channel 1
    d[:, 0], x[:, 0] = 0, 0
    d[r, 0], x[c, 0] = SUMS[kind]
    w = torch.zeros((co, 2, ci, 2, lg.K), device="cuda")

    def run():
        _, dw, _ = layers.lsc_backward(lg, x, w, d, ci, co, need_input=False)
        L.check_device_error(kind)
        return dw

    dw = run()
    L.set_tensor_cores(False)
    try:
        ref = run()
    finally:
        L.set_tensor_cores(True)
    hit = torch.zeros(w.shape, dtype=torch.bool, device="cuda")
    if kind == "nan":  # a NaN in dY meets every row of X
        hit[11, 1] = True
    else:
        hit[11, 1, 1, 0] = True
    assert bool(torch.isfinite(ref[~hit]).all()) and bool(torch.isfinite(ref[hit]).all()) == ("large" in kind)
    assert torch.equal(torch.isnan(dw), torch.isnan(ref))
    assert torch.equal(torch.isposinf(dw), torch.isposinf(ref)) and torch.equal(torch.isneginf(dw), torch.isneginf(ref))
    for part in (hit, ~hit):
        a, b = dw[part].double(), ref[part].double()
        if bool(torch.isfinite(b).all()):
            assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) <= 2e-6
