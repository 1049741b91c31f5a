"""The tensor-core build of the collapsed operator at the edges of its tiles: against the FP64
collapse of the library's own FP32 tables, each entry within one BF16 ulp plus the bound of an
FP32 sum of K products, (K + 1) 2^-24 sum_k |w_k| |M_k| (as test_gpu_build_w derives it); zero
outside the shell window.  The weights start one float off a 16-byte boundary."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    # four output channels per tile, a short last tile
    "ci32": dict(m=[30, 30], order_in=8, order=8, ci=32, co=7, R=2, Sec=6, win="adjacent"),
    # 64 -> 64 channels, three shells: M images change inside a CTA's run of tiles
    "hidden": dict(m=[30, 30, 30], order_in=8, order=8, ci=64, co=64, R=4, Sec=12, win="adjacent"),
    # 28 input coefficients (9 rows of 28 per tile), one kernel step (K = 6)
    "order6": dict(m=[30, 30, 30], order_in=6, order=6, ci=8, co=5, R=1, Sec=5, win="same"),
    # one coefficient in: all rows in one tile; 128 input channels
    "order0_in": dict(m=[40], order_in=0, order=8, ci=128, co=3, R=1, Sec=3, win="all"),
    # 91 output rows of 91 entries: two rows per tile, an odd last row; K = 64
    "order12": dict(m=[100], order_in=12, order=12, ci=8, co=2, R=7, Sec=9, win="same"),
    # one input shell into three output shells
    "one_to_three": dict(m=[30, 30, 30], s_in=1, order_in=4, order=8, ci=16, co=9, R=2, Sec=6, win="all"),
}


@pytest.mark.parametrize("case", list(CASES))
def test_tiles_of_the_operator_build(case):
    cfg = CASES[case]
    S, ci, co = len(cfg["m"]), cfg["ci"], cfg["co"]
    s_in = cfg.get("s_in", S)
    dirs, bvals = synth.multishell_table(cfg["m"], [1000, 2000, 3000][:S], seed=35)
    lb = L.SHBasis(dirs, bvals, cfg["order"], 0.006)
    lg = L.LSCGeometry(lb, cfg["order_in"], s_in, np.deg2rad(25), cfg["R"], cfg["Sec"], cfg["win"])
    K, n_in, n_out, V = lg.K, lg.n_in, lg.n_out, 64
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    flat = 0.1 * torch.randn(1 + co * S * ci * s_in * K, generator=gen, device="cuda")
    w = flat[1:].view(co, S, ci, s_in, K)
    x = layers.as_act(torch.zeros((s_in * ci * n_in, V), dtype=torch.bfloat16, device="cuda"))
    t, ptr, _ = ws = layers.lsc_workspace(lg, V, ci, co, torch.bfloat16, False)
    t.fill_(0xFF)  # every entry of W has to be written
    L.trace_enable(True)
    try:
        layers.lsc_forward(lg, x, w, None, ci, co, workspace=ws)
        torch.cuda.synchronize()
        assert "lsc_build_w_tc" in L.trace_summary()
    finally:
        L.trace_enable(False)
    L.check_device_error("operator build")
    rows, ld = S * co * n_out, s_in * ci * n_in
    off = ptr - t.data_ptr()
    W = t[off:off + rows * ld * 2].view(torch.bfloat16).double().view(S, co, n_out, s_in, ci, n_in)
    for s in range(S):
        tab = lg.tables(s)
        M = torch.from_numpy(tab["M"].astype(np.float32).astype(np.float64)).cuda()
        for p in range(s_in):
            got = W[s, :, :, p]
            if not tab["window"][p]:
                assert bool((got == 0).all())
                continue
            wd = w[:, s, :, p].double()
            ref = torch.einsum("ock,kab->oacb", wd, M)
            err = (K + 1) * 2.0 ** -24 * torch.einsum("ock,kab->oacb", wd.abs(), M.abs())
            ref16 = ref.bfloat16().double()
            ulp = torch.exp2(torch.floor(torch.log2(torch.maximum(ref16.abs(), got.abs()).clamp_min(1e-30)))) * 2.0 ** -7
            assert bool(((got - ref16).abs() <= ulp + err).all()), (s, p)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("m,s_in,order_in,order,ci,co,R,Sec,win", [
    ([40, 40, 40], 1, 4, 8, 1, 64, 4, 12, "all"),      # the network's first layer: one padding column
    ([40], 1, 8, 8, 3, 5, 3, 8, "same"),               # a last group of three pairs
    ([40, 40, 40], 3, 4, 6, 8, 3, 6, 13, "adjacent"),  # K = 79: two chunks, and shells outside the window
    ([1], 1, 0, 0, 1, 1, 1, 1, "all"),
])
def test_small_operator_equals_the_blocked_build(m, s_in, order_in, order, ci, co, R, Sec, win, dtype):
    dirs, bvals = synth.multishell_table(m, [1000, 2000, 3000][:len(m)], seed=36)
    lb = L.SHBasis(dirs, bvals, order, 0.006 if order else 0.0)
    lg = L.LSCGeometry(lb, order_in, s_in, np.deg2rad(25), R, Sec, win)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    w = torch.randn((co, len(m), ci, s_in, lg.K), generator=gen, device="cuda")
    b = torch.randn((co, len(m)), generator=gen, device="cuda")
    x = layers.as_act(torch.zeros((s_in * ci * lg.n_in, 64), dtype=dtype, device="cuda"))
    rows, ld = len(m) * co * lg.n_out, s_in * ((ci * lg.n_in + 7) // 8 * 8)
    Ws, ys = [], []
    for mode in (L.TC_PREFER, L.TC_OFF):  # without tensor cores the forward reads Wt: the blocked kernel writes both
        t, ptr, _ = ws = layers.lsc_workspace(lg, 64, ci, co, dtype, False)
        t.fill_(0xFF)
        L.set_tensor_cores(mode)
        try:
            ys.append(layers.lsc_forward(lg, x, w, b, ci, co, workspace=ws))
        finally:
            L.set_tensor_cores(True)
        off = ptr - t.data_ptr()
        Ws.append(t[off:off + rows * ld * x.element_size()].view(dtype).clone())
    L.check_device_error("operator build")
    assert torch.equal(Ws[0], Ws[1]) and bool(torch.isfinite(Ws[0]).all())
    assert torch.equal(ys[0], ys[1])  # x is zero: the bias alone
