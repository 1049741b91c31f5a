"""Which kernel makes the weight gradient's reduction: the trace tells the tensor-core one from the
CUDA cores', and both agree.

Tolerance of the relative L2 difference: each side's sum is within n 2^-24 of FP64, n the additions
at full magnitude, at most 30 here for the two together (16 voxels): 2e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu

# (directions, order in, order out, input shells, rings, sectors, window, resampling-free, c_in, c_out, dtype, tensor cores)
CASES = {
    "hidden": ([40, 40, 40], 8, 8, 3, 4, 12, "adjacent", False, 64, 64, "bf16", True),
    "first_layer": ([40, 40, 40], 4, 8, 1, 4, 12, "all", False, 1, 64, "bf16", True),
    "k64": ([40, 40], 8, 8, 2, 7, 9, "all", False, 5, 48, "bf16", True),
    "co130": ([40, 40], 8, 8, 2, 2, 6, "same", False, 3, 130, "bf16", True),
    "resampling_free": ([40, 40, 40], 8, 8, 3, 2, 6, "adjacent", True, 8, 12, "bf16", True),
    # 120 output coefficients: eight k-steps of one input coefficient
    "order14": ([128], 4, 14, 1, 2, 6, "same", False, 4, 20, "bf16", True),
    "64_to_4": ([40, 40], 8, 8, 2, 2, 6, "adjacent", False, 64, 4, "bf16", True),
    "16_to_1": ([40, 40], 8, 8, 2, 2, 6, "adjacent", False, 16, 1, "bf16", True),
    # more than 32 short runs a step
    "64_to_1": ([40, 40], 8, 8, 2, 2, 6, "adjacent", False, 64, 1, "bf16", False),
    "33_to_3": ([40, 40], 8, 8, 2, 2, 6, "adjacent", False, 33, 3, "bf16", False),
    # more than 64 kernel points
    "k73": ([40, 40], 8, 8, 2, 6, 12, "adjacent", False, 3, 5, "bf16", False),
    # the M images of 45 input coefficients in one part: more than a CTA's shared memory
    "order8_to_0": ([40], 8, 0, 1, 2, 6, "same", False, 4, 8, "bf16", False),
    # 45 x 120 coefficients
    "order8_to_14": ([128], 8, 14, 1, 2, 6, "same", False, 4, 8, "bf16", False),
    "f32": ([40, 40], 8, 8, 2, 2, 6, "adjacent", False, 8, 8, "f32", False),
}


@pytest.mark.parametrize("case", list(CASES))
def test_route_and_agreement(case):
    m, order_in, order, s_in, rings, sectors, win, free, ci, co, dt, tc = CASES[case]
    S, V = len(m), 16
    dirs, bvals = synth.multishell_table(m, [1000, 2000, 3000][:S], seed=33)
    lb = L.SHBasis(dirs, bvals, order, 0.006 if order else 0.0)
    lg = L.LSCGeometry(lb, order_in, s_in, np.deg2rad(25), rings, sectors, win, neighbours=free)
    dtype = torch.bfloat16 if dt == "bf16" else torch.float32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x = torch.randn((s_in * ci * lg.n_in, V), generator=gen, device="cuda").to(dtype)
    d = torch.randn((S * co * lg.n_out, V), generator=gen, device="cuda").to(dtype)
    w = torch.zeros((co, S, ci, s_in, lg.K), device="cuda")

    def run():
        L.trace_enable(True)
        try:
            _, dw, db = layers.lsc_backward(lg, x, w, d, ci, co, need_input=False)
            torch.cuda.synchronize()
            names = {n for n in L.trace_summary() if n.startswith("lsc_reduce_dw")}
        finally:
            L.trace_enable(False)
        L.check_device_error(case)
        return dw.double(), db.double(), names

    dw, db, names = run()
    assert names == ({"lsc_reduce_dw_tc"} if tc else {"lsc_reduce_dw"})
    L.set_tensor_cores(False)
    try:
        dw0, db0, names = run()
    finally:
        L.set_tensor_cores(True)
    assert names == {"lsc_reduce_dw"}
    for a, b in ((dw, dw0), (db, db0)):
        assert float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b)) <= 2e-6
