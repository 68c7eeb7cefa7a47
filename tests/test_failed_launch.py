"""A launch that CUDA refuses fails its own call and no later one.  The refusal is
made on the host: a stream whose capture a forbidden call has invalidated takes
no launch, and nothing reaches the GPU."""
import ctypes

import numpy as np
import pytest

from paper_2604_06602_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class _Stream:
    """A stream made with the driver API; `cuda_stream` is its handle."""

    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        h = ctypes.c_void_p()
        assert self.cu.cuStreamCreate(ctypes.byref(h), 1) == 0  # non-blocking
        self.cuda_stream = h.value

    def spoil_capture(self):
        h = ctypes.c_void_p(self.cuda_stream)
        assert self.cu.cuStreamBeginCapture_v2(h, 1) == 0       # this thread's calls
        assert self.cu.cuStreamSynchronize(h) != 0              # not allowed while capturing

    def end_capture(self):
        graph = ctypes.c_void_p()
        h = ctypes.c_void_p(self.cuda_stream)
        assert self.cu.cuStreamEndCapture(h, ctypes.byref(graph)) != 0
        assert self.cu.cuStreamDestroy_v2(h) == 0


@pytest.mark.parametrize("call", ["one", "noalloc", "segmented"])
def test_the_next_calls_succeed(call):
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    x = torch.from_numpy(synth.random_curve(5, 6000, nan_runs=2, run_len=(1, 200))).cuda()
    off, W = np.array([0, 2500, 6000], np.int64), np.array([25, 25], np.int32)

    def run(stream=None):
        if call == "one":
            return umi.detrend(x, 25, stream=stream)[0]
        if call == "noalloc":
            return umi.detrend_batched_noalloc(x, off, W, stream=stream)[0]
        return umi.detrend_segmented(x, off, W, stream=stream)[0]

    want = run()
    seg = umi.detrend_segmented(x, off, W)[0]
    torch.cuda.synchronize()
    s = _Stream()
    s.spoil_capture()
    try:
        with pytest.raises(umi.UmiError) as e:
            run(stream=s)
        assert e.value.status == umi.UMI_ERR_CUDA
    finally:
        s.end_capture()
    # Segmented first: it asks CUDA for the thread's last error after its own launches.
    got_seg = umi.detrend_segmented(x, off, W)[0]
    got = run()
    torch.cuda.synchronize()
    assert torch.equal(got_seg.view(torch.int32), seg.view(torch.int32))
    assert torch.equal(got.view(torch.int32), want.view(torch.int32))
