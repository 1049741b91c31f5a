"""FP32 transforms on the tensor cores where their rings wrap: many tiles per CTA, even and odd numbers
of A stages and of chunks per tile, outputs in one accumulator and in two halves, read through TMA and,
where the rows start on no 16-byte boundary, as they lie (the call itself, not the copy that the
layers fall back to): against the FP64 operators, and the two forms of input bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import sh as osh  # noqa: E402
from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402
from tests._layout import TOL_BF16, TOL_F32  # noqa: E402

pytestmark = pytest.mark.gpu

# directions per shell, order, channels, voxels (4 k + 1 or 3: unaligned rows)
SHAPES = {
    # five A stages (two accumulators of 128 columns), two chunks of 45 rows; four chunks of 120 rows
    "120": ([120], 8, 1, 300001),
    # three chunks per tile of a fit; six A stages
    "90": ([90], 8, 1, 300001),
    # two accumulators of three blocks (64 outputs), two A stages
    "64_order6": ([64], 6, 2, 100003),
    # halves: 128 and 128, 128 and 96 columns, a shell of one half beside them
    "256": ([256], 8, 1, 100003),
    "209": ([209], 4, 2, 60001),
    "mixed": ([240, 128, 16], 4, 1, 60001),
    "256_few": ([256], 8, 3, 131),
    # the most outputs that fit two whole accumulators
    "208": ([208], 4, 1, 100003),
}


@pytest.mark.parametrize("kind", list(layers._TRANSFORMS))
@pytest.mark.parametrize("shape", list(SHAPES))
def test_against_fp64_and_the_aligned_form(shape, kind):
    m, order, C, V = SHAPES[shape]
    dirs, bvals = synth.multishell_table(m, [1000, 2000, 3000][:len(m)], seed=51)
    ob = osh.SHBasisOracle(dirs, bvals, order, 0.006)
    lb = L.SHBasis(dirs, bvals, order, 0.006)
    from_sig = kind in ("signal2sh", "sh2signal_backward")
    S, N = lb.n_shells, lb.n_coef
    rows_in, rows_out = (C * sum(m), S * C * N) if from_sig else (S * C * N, C * sum(m))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    x = torch.randn((rows_in, V), generator=gen, device="cuda")
    copy = layers.empty_act(rows_in, V, torch.float32).copy_(x)
    ops = {"signal2sh": [P for P in ob.P], "sh2signal": [B for B in ob.B],
           "signal2sh_backward": [P.T for P in ob.P], "sh2signal_backward": [B.T for B in ob.B]}[kind]
    for out_t, tol in ((torch.float32, TOL_F32), (torch.bfloat16, TOL_BF16)):
        want = layers.transform(kind, lb, copy, C, out_t)
        got = layers.empty_act(rows_out, V, out_t)
        st = L.get().delimit_transform_unaligned(lb.handle, layers._KINDS[kind], x.data_ptr(), got.data_ptr(), V, C, V,
                                                 got.stride(0), L.F32, layers._code(got),
                                                 torch.cuda.current_stream().cuda_stream)
        assert st == L.OK
        L.check_device_error(kind)
        assert torch.equal(got, want)
        r0 = o0 = 0
        for T in ops:  # rows (shell, channel, feature)
            T = torch.from_numpy(np.ascontiguousarray(T)).cuda()
            n_out, n_in = T.shape
            for c in range(C):
                ref = T @ x[r0:r0 + n_in].double()
                err = want[o0:o0 + n_out].double() - ref
                assert float(torch.linalg.vector_norm(err) / torch.linalg.vector_norm(ref)) <= tol, (c, out_t)
                r0, o0 = r0 + n_in, o0 + n_out
