"""The device filter after a call that failed on the same thread: a call on a
stream that is being captured fails in its wait for the stream and leaves CUDA's
error pending.  The next ordinary call must neither take that error for its
own launch's nor return before its kernel has stored the count."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

vx = pytest.importorskip("paper_2502_09541_gb300")
torch = pytest.importorskip("torch")

THREAD_LOCAL = 1  # CU_STREAM_CAPTURE_MODE_THREAD_LOCAL


@pytest.mark.parametrize("n", [10_007, 3_000_001])
def test_call_after_a_failed_capture(n):
    v = torch.arange(n, dtype=torch.int32, device="cuda") % 100
    out = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    preds = [(0, vx.VX_LT, 7, 0)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(handle, THREAD_LOCAL) == 0
    try:
        with pytest.raises(RuntimeError):
            vx.vx_filter_device_static([v.data_ptr()], preds, n, 0, out.data_ptr(), n, stream.cuda_stream)
    finally:
        assert cu.cuStreamEndCapture(handle, ctypes.byref(graph)) != 0  # the wait ended the capture
    torch.cuda.synchronize()
    assert (out == -1).all()  # nothing ran
    want = np.nonzero(v.cpu().numpy() < 7)[0]
    for _ in range(2):
        st, cnt = vx.vx_filter_device_static([v.data_ptr()], preds, n, 0, out.data_ptr(), n)
        assert st == vx.VX_OK and cnt == len(want)
        assert np.array_equal(out[:cnt].cpu().numpy(), want)
