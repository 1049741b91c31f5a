"""The error of the weight gradient's reduction on the tensor cores (BF16 activations, K <= 64):
no larger than that of the FP32 sum on the CUDA cores.

16 voxels, so that the voxel sums (one MMA chunk) leave the reduction's error to be seen.  Two
bounds, both of the relative L2 error against FP64.  From the additions at full magnitude, each
within 2^-24 of the sum: two k-steps in one accumulator, the accumulators of a part and its small
products, the parts, four for the voxel sums.  And the CUDA cores' own
error on the same inputs plus one such rounding.  (All six part products in one accumulator: 1.1e-6 to 2.1e-6, against 1.5e-7 to 1.8e-7
on the CUDA cores.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lsc as olsc  # noqa: E402
from oracle import sh as osh  # noqa: E402
from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    "64_to_64": dict(m=[40, 40, 40], ci=64, co=64, R=4, Sec=12, win="adjacent"),
    "1_to_64": dict(m=[40, 40, 40], ci=1, co=64, order_in=4, s_in=1, R=4, Sec=12, win="all"),
    # one k-step per input coefficient; five and six of them
    "order4": dict(m=[40], ci=8, co=16, order_in=4, order=4, win="same"),
    "order10": dict(m=[90], ci=16, co=16, order_in=10, order=10, win="same"),
    "order12_from2": dict(m=[100], ci=4, co=20, order_in=2, order=12, win="same"),
}


@pytest.mark.parametrize("case", list(CASES))
def test_error_not_above_the_fp32_sum(case):
    cfg = dict(order_in=8, order=8, R=2, Sec=6)
    cfg.update(CASES[case])
    S, ci, co, V = len(cfg["m"]), cfg["ci"], cfg["co"], 16
    s_in = cfg.get("s_in", S)
    dirs, bvals = synth.multishell_table(cfg["m"], [1000, 2000, 3000][:S], seed=33)
    geo = (cfg["order_in"], s_in, np.deg2rad(25), cfg["R"], cfg["Sec"], cfg["win"])
    og = olsc.LSCOracle(osh.SHBasisOracle(dirs, bvals, cfg["order"], 0.006), *geo)
    lb = L.SHBasis(dirs, bvals, cfg["order"], 0.006)
    lg = L.LSCGeometry(lb, *geo)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x = torch.randn((s_in * ci * lg.n_in, V), generator=gen, device="cuda").bfloat16()
    d = torch.randn((S * co * lg.n_out, V), generator=gen, device="cuda").bfloat16()
    w = torch.zeros((co, S, ci, s_in, lg.K), device="cuda")
    xs, ds = x.double().reshape(s_in, ci * lg.n_in, V), d.double().reshape(S, co * lg.n_out, V)
    ref = torch.zeros(w.shape, dtype=torch.float64, device="cuda")
    for s in range(S):
        for p in range(s_in):
            if og.win[s, p]:
                mats = torch.from_numpy(np.ascontiguousarray(og.pair_mats(s, p))).cuda()
                ref[:, s, :, p] = torch.einsum("kab,oaib->oik", mats,
                                               (ds[s] @ xs[p].T).reshape(co, lg.n_out, ci, lg.n_in))

    def error():
        _, dw, _ = layers.lsc_backward(lg, x, w, d, ci, co, need_input=False)
        L.check_device_error(case)
        return float(torch.linalg.vector_norm(dw.double() - ref) / torch.linalg.vector_norm(ref))

    tc = error()
    L.set_tensor_cores(False)
    try:
        cc = error()
    finally:
        L.set_tensor_cores(True)
    parts = -(-lg.n_in * lg.n_out // 256)
    steps = -(-lg.n_in // parts) * -(-lg.n_out // 16)
    sums = 2 + -(-steps // 2) + 1 + parts + 4
    assert tc <= sums * 2.0 ** -24, (tc, cc)
    assert tc <= cc + 2.0 ** -24, (tc, cc)
