"""Transforms of FP32 inputs whose rows start on no 16-byte boundary, read as they lie: bit for bit
the result of the padded copy (the same tiles, products and sums), over every offset, the four
transforms, output types, ragged tiles, several channels and shells, and more than 128 outputs."""
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = {"3x40": ([40, 33, 20], 6, 2), "30_order4": ([30], 4, 1), "150": ([150], 8, 1), "1": ([1], 0, 3)}


@pytest.mark.parametrize("kind", list(layers._TRANSFORMS))
@pytest.mark.parametrize("shape", list(SHAPES))
def test_unaligned_input_equals_its_copy(shape, kind):
    m, order, C = SHAPES[shape]
    dirs, bvals = synth.multishell_table(m, [1000, 2000, 3000][:len(m)], seed=51)
    lb = L.SHBasis(dirs, bvals, order, 0.006 if order else 0.0)
    from_sig = kind in ("signal2sh", "sh2signal_backward")
    rows = C * lb.n_dirs if from_sig else lb.n_shells * C * lb.n_coef
    for n_vox, off in ((1, 1), (127, 0), (130, 3), (1001, 2), (4099, 1)):
        buf = torch.randn(rows * n_vox + off, device="cuda")
        x = buf[off:].view(rows, n_vox)
        copy = layers.empty_act(rows, n_vox, torch.float32)
        copy.copy_(x)
        for out_t in (torch.float32, torch.bfloat16):
            want = layers.transform(kind, lb, copy, C, out_t)
            got = layers.transform(kind, lb, x, C, out_t)
            L.check_device_error(kind)
            assert torch.equal(got, want), (n_vox, off, out_t)


def test_volume_tensor_and_refusals():
    dirs, bvals = synth.multishell_table([30], [1000], seed=52)
    layer = layers.Signal2SH(4, dirs, 0.006)
    vol = torch.rand((1, 30, 7, 9, 11), device="cuda")  # 693 voxels
    got = layer(vol)
    flat = layers.empty_act(30, 693, torch.float32)
    flat.copy_(vol.reshape(30, 693))
    want = layers.transform("signal2sh", layer.basis, flat, 1)
    assert got.shape == (1, 15, 7, 9, 11) and torch.equal(got.reshape(15, 693), want)
    # the aligned entry keeps its rule, and without tensor cores the copy is made
    x, lib = vol.reshape(30, 693), L.get()
    out = layers.empty_act(15, 693, torch.float32)
    st = torch.cuda.current_stream().cuda_stream
    args = (x.data_ptr(), out.data_ptr(), 693, 1, 693, out.stride(0))
    assert lib.delimit_signal2sh(layer.basis.handle, *args, L.F32, L.F32, st) == L.ERR_ALIGNMENT
    assert lib.delimit_transform_unaligned(layer.basis.handle, 0, *args, L.BF16, L.F32, st) == L.ERR_UNSUPPORTED
    L.set_tensor_cores(False)
    try:
        assert lib.delimit_transform_unaligned(layer.basis.handle, 0, *args, L.F32, L.F32, st) == L.ERR_UNSUPPORTED
        ref = layers.transform("signal2sh", layer.basis, x, 1)
    finally:
        L.set_tensor_cores(True)
    assert torch.allclose(ref, want, rtol=0, atol=1e-5)
