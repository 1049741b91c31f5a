"""Gathered Signal2SH over the widths of its outputs (15, 28, 45 and 66 coefficients: a kernel of its
own for each of the first three, two chunks of outputs for the last), both input and both output
types, channels and shells, against the FP64 oracle's operators."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sh as osh  # noqa: E402
from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402
from tests._layout import TOL_BF16, TOL_F32  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("out_t", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("in_t", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("order,m,n", [(4, [30, 20], 3001), (6, [45, 60], 3001), (8, [64, 50], 3001),
                                       (8, [64, 50], 20011), (8, [70, 90], 20011), (10, [70, 90], 3001),
                                       (10, [128], 130), (8, [45], 1)])
def test_against_the_oracle(order, m, n, in_t, out_t):
    C, n_src = 2, 2 * n + 37
    dirs, bvals = synth.multishell_table(m, [1000, 2000][:len(m)], seed=61)
    ob = osh.SHBasisOracle(dirs, bvals, order, 0.006)
    lb = L.SHBasis(dirs, bvals, order, 0.006)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(9)
    vol = layers.empty_act(C * sum(m), n_src, in_t)
    vol.copy_(torch.rand(vol.shape, generator=gen, device="cuda").add_(0.1).to(in_t))
    b0 = torch.rand(n_src, generator=gen, device="cuda") + 0.5
    b0[::17] = 0.0
    index = torch.randperm(n_src, generator=gen, device="cuda")[:n].sort().values
    got = layers.signal2sh_gather(lb, vol, index, b0=b0, channels=C, out_dtype=out_t)
    L.check_device_error("gather")
    b = b0[index].double()
    x = torch.where(b > 0, vol[:, index].double() / b, torch.zeros((), dtype=torch.float64, device="cuda"))
    ref, row = [], 0
    for s, k in enumerate(m):  # rows (shell, channel, direction) -> (shell, channel, coefficient)
        P = torch.from_numpy(np.ascontiguousarray(ob.P[s])).cuda()
        ref.append((P @ x[row:row + C * k].reshape(C, k, n)).reshape(-1, n))
        row += C * k
    ref = torch.cat(ref)
    assert got.dtype == out_t and got.shape == ref.shape
    err = float(torch.linalg.vector_norm(got.double() - ref) / torch.linalg.vector_norm(ref))
    assert err <= (TOL_F32 if out_t == torch.float32 else TOL_BF16)
