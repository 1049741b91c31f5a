"""The weight gradient's last step on the tensor cores (BF16 activations, K <= 64), at the
edges of its tiles, against FP64.

dw[co,s,ci,s',k] = sum_ab M_{s,s'}[k][a][b] sum_v dY[(s,co,a),v] X[(s',ci,b),v] from the BF16
values that the GEMMs read, so only FP32 sums separate the two.  Tolerance: the voxel sum adds
V / 16 MMAs into one FP32 accumulator (per voxel split), the reduction at most about 110 (18 per
input coefficient, one part of the range); a sum of n MMAs is within n 2^-24 of the terms' size,
(300 / 16 + 110) 2^-24 = 8e-6 at 300 voxels: 2e-5.  Over 4,096 voxels the voxel sum dominates:
the bound that the full-size test of the weight gradient takes, 2e-4.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import lsc as olsc  # noqa: E402
from oracle import sh as osh  # noqa: E402
from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    # one output channel: 128 input channels per tile, the last tile short
    "co1": dict(m=[40, 40], ci=130, co=1, win="adjacent"),
    # runs that start off the 16-byte grid (7 x 45 rows per shell), a short last tile
    "co7": dict(m=[40, 40, 40], ci=20, co=7, win="adjacent"),
    # 48 of 64 rows per input channel, K = 64 exactly
    "co48_k64": dict(m=[40, 40], ci=5, co=48, R=7, Sec=9, win="all"),
    # more than 128 output channels: a full and a short chunk per input channel
    "co130": dict(m=[40, 40], ci=3, co=130, win="same"),
    # 64 -> 64 channels: many units per CTA, the parts' images change under way
    "hidden": dict(m=[40, 40, 40], ci=64, co=64, R=4, Sec=12, win="adjacent"),
    # 28 output coefficients (an even row length), 15 input coefficients
    "order6_from4": dict(m=[40, 40], ci=9, co=6, order_in=4, order=6, win="adjacent"),
    # one k-step per input coefficient; one input shell into three
    "first_layer": dict(m=[40, 40, 40], ci=1, co=64, order_in=4, s_in=1, win="all"),
    # 91 output coefficients (six k-steps), 6 input coefficients
    "order12": dict(m=[100], ci=4, co=20, order_in=2, order=12, win="same"),
    # images per shell pair
    "resampling_free": dict(m=[40, 40, 40], ci=8, co=12, win="adjacent", neighbours=True),
    # several voxel splits
    "splits": dict(m=[40, 40], ci=3, co=5, win="adjacent", V=16390, tol=2e-4),
    # K = 73: the CUDA-core reduction
    "k73": dict(m=[40, 40], ci=3, co=5, R=6, Sec=12, win="adjacent"),
}


@pytest.mark.parametrize("case", list(CASES))
def test_weight_gradient_against_fp64(case):
    cfg = dict(order_in=8, order=8, R=2, Sec=6, V=300, tol=2e-5)
    cfg.update(CASES[case])
    S, ci, co, V = len(cfg["m"]), cfg["ci"], cfg["co"], cfg["V"]
    s_in = cfg.get("s_in", S)
    dirs, bvals = synth.multishell_table(cfg["m"], [1000, 2000, 3000][:S], seed=33)
    ob = osh.SHBasisOracle(dirs, bvals, cfg["order"], 0.006)
    rad, free = np.deg2rad(25), cfg.get("neighbours", False)
    cls = olsc.LSCNeighbourOracle if free else olsc.LSCOracle
    og = cls(ob, cfg["order_in"], s_in, rad, cfg["R"], cfg["Sec"], cfg["win"])
    lb = L.SHBasis(dirs, bvals, cfg["order"], 0.006)
    lg = L.LSCGeometry(lb, cfg["order_in"], s_in, rad, cfg["R"], cfg["Sec"], cfg["win"], neighbours=free)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    x = layers.as_act(torch.randn((s_in * ci * lg.n_in, V), generator=gen, device="cuda").bfloat16())
    d = layers.as_act(torch.randn((S * co * lg.n_out, V), generator=gen, device="cuda").bfloat16())
    w = torch.zeros((co, S, ci, s_in, lg.K), device="cuda")
    _, dw, db = layers.lsc_backward(lg, x, w, d, ci, co, need_input=False)
    L.check_device_error("backward")
    xs, ds = x.double().reshape(s_in, ci * lg.n_in, V), d.double().reshape(S, co * lg.n_out, V)
    ref, mats = torch.zeros_like(dw, dtype=torch.float64), None
    for s in range(S):
        for p in range(s_in):
            if og.win[s, p]:
                mats = torch.from_numpy(np.ascontiguousarray(og.pair_mats(s, p))).cuda()
                G = (ds[s] @ xs[p].T).reshape(co, lg.n_out, ci, lg.n_in)
                ref[:, s, :, p] = torch.einsum("kab,oaib->oik", mats, G)
    q = torch.stack([torch.from_numpy(og.Pout[s].sum(1)).cuda() for s in range(S)])
    ref_db = torch.einsum("soa,sa->os", ds.reshape(S, co, lg.n_out, V).sum(-1), q)
    rel = lambda a, b: float(torch.linalg.vector_norm(a.double() - b) / torch.linalg.vector_norm(b))  # noqa: E731
    errs = {"dw": rel(dw, ref), "db": rel(db, ref_db)}
    assert all(e <= cfg["tol"] for e in errs.values()), errs
    out = ~torch.from_numpy(og.win).cuda()
    assert bool((dw.permute(1, 3, 0, 2, 4)[out] == 0).all())
