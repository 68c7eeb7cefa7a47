"""One-curve calls and the allocation-free batched call captured into a CUDA
graph by the caller: launches that follow each other on the captured stream
keep their order (each output is checked on replay with new inputs), and give
the bits of the plain calls."""
import numpy as np
import pytest

from paper_2604_06602_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_captured_calls_replay_on_new_inputs():
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    xs = [torch.from_numpy(synth.random_curve(300 + k, 9000, nan_runs=2, run_len=(1, 300))).cuda() for k in range(3)]
    off = np.array([0, 2500, 9000], np.int64)
    Ws = np.array([25, 361], np.int32)
    x = xs[0].clone()
    bufs = [torch.empty_like(x) for _ in range(8)]

    def chain():
        # Each call reads what the one before wrote.
        umi.detrend(x, 361, trend=bufs[0], detr=bufs[1])
        umi.detrend(bufs[1], 25, trend=bufs[2], detr=bufs[3])
        umi.detrend_batched_noalloc(bufs[3], off, Ws, trend=bufs[4], detr=bufs[5])
        umi.detrend(bufs[5], 721, trend=bufs[6], detr=bufs[7])

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        chain()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        chain()
    for v in xs[1:]:
        x.copy_(v)
        chain()
        torch.cuda.synchronize()
        want = [b.clone() for b in bufs]
        for b in bufs:
            b.fill_(-1.0)
        g.replay()
        torch.cuda.synchronize()
        for b, w in zip(bufs, want):
            assert torch.equal(b.view(torch.int32), w.view(torch.int32))
