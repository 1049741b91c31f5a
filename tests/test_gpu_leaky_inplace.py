"""The leaky ReLU and its backward in place (y = x, dx = dy) against buffers of their own: the same bits."""
import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,n", [(3, 1), (45, 1001), (7, 65536)])
def test_in_place(rows, n, dtype):
    lib, code, st = L.get(), layers._DT[dtype], torch.cuda.current_stream().cuda_stream
    y = layers.as_act(torch.randn((rows, n), device="cuda").to(dtype))
    dy = layers.as_act(torch.randn((rows, n), device="cuda").to(dtype))
    want = [layers.empty_act(rows, n, dtype) for _ in range(2)]
    ld = y.stride(0)

    def run(x_out, dx):
        assert lib.delimit_leaky_relu_backward(y.data_ptr(), dy.data_ptr(), dx.data_ptr(), rows, n, ld, dy.stride(0),
                                               dx.stride(0), 0.1, code, st) == L.OK
        assert lib.delimit_leaky_relu(y.data_ptr(), x_out.data_ptr(), rows, n, ld, x_out.stride(0), 0.1, code, st) == L.OK

    run(*want)
    run(y, dy)
    assert torch.equal(y, want[0]) and torch.equal(dy, want[1])
