"""A call that fails reports its own error and leaves none behind for the next."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def test_a_failed_launch_is_reported_once():
    """Launches into a stream capture that a synchronisation has ended fail, each with its error; after the capture the
    next call runs."""
    import torch
    import paper_2006_10091_gb300 as he
    stream = torch.cuda.Stream()
    ctx = he.Context(12, 3, 40, 1, 60, 2.0 ** 30, seed=3, stream=stream.cuda_stream)
    with torch.cuda.stream(stream):
        a, out = ctx.new_ct(3), ctx.new_ct(3)
        a.tensor.zero_()
        a.level, a.scale = 3, 2.0 ** 30
    he.he_autotune(ctx, 2, 1)
    he.he_add(ctx, a, a, out)
    torch.cuda.synchronize()
    cuda = ctypes.CDLL("libcuda.so.1")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert cuda.cuStreamBeginCapture_v2(handle, 1) == 0  # CU_STREAM_CAPTURE_MODE_THREAD_LOCAL
    try:
        with pytest.raises(he.HeError):
            he.he_sync(ctx)                              # not allowed while capturing: the capture is invalid now
        with pytest.raises(he.HeError):
            he.he_add(ctx, a, a, out)
    finally:
        cuda.cuStreamEndCapture(handle, ctypes.byref(graph))
    he.he_autotune(ctx, 2, 1)                            # (checks its first launch by cudaGetLastError)
    he.he_add(ctx, a, a, out)
    he.he_sync(ctx)
