"""A call made as a host thread's first CUDA work (autograd's backward thread makes such calls):
the thread has no current context yet, and the results are those of the main thread."""
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_1808_01517_gb300 import _lib as L  # noqa: E402
from paper_1808_01517_gb300 import layers, synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("call", ["transform", "lsc_backward"])
def test_first_cuda_call_of_a_thread(call, dtype):
    dirs, bvals = synth.multishell_table([30], [1000], seed=5)
    lb = L.SHBasis(dirs, bvals, 4, 0.006)
    lg = L.LSCGeometry(lb, 4, 1, 0.4, 1, 5, "same")
    x = layers.as_act(torch.randn((2 * 15, 500), device="cuda").to(dtype))
    d = layers.as_act(torch.randn((3 * 15, 500), device="cuda").to(dtype))
    s = layers.as_act(torch.randn((30, 500), device="cuda").to(dtype))
    w = torch.randn((3, 1, 2, 1, lg.K), device="cuda")
    out = layers.empty_act(15, 500, dtype)
    ws = layers.lsc_workspace(lg, 500, 2, 3, dtype, True)
    dw = torch.empty_like(w)
    st = torch.cuda.current_stream().cuda_stream
    code = layers._code(x)

    def run():  # raw calls on buffers that exist: nothing else touches CUDA in the thread
        if call == "transform":
            L.check(L.get().delimit_signal2sh(lb.handle, s.data_ptr(), out.data_ptr(), 500, 1, s.stride(0),
                                              out.stride(0), code, code, st), call)
        else:
            L.check(L.get().delimit_lsc_backward(lg.handle, x.data_ptr(), w.data_ptr(), d.data_ptr(), None,
                                                 dw.data_ptr(), None, 500, 2, 3, x.stride(0), d.stride(0), code, 0,
                                                 ws[1], ws[2], st), call)

    run()
    want = (out if call == "transform" else dw).clone()
    out.zero_(), dw.zero_()
    torch.cuda.synchronize()
    failed = []

    def guarded():
        try:
            run()
        except Exception as e:  # noqa: BLE001
            failed.append(e)

    t = threading.Thread(target=guarded)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    assert torch.equal(out if call == "transform" else dw, want)
