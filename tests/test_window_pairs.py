"""The 32-lane variant of 12 slots finishes its windows in pairs: odd and even
chains, curves that end inside a pair, pairs of which one or both windows give
no output, both forms of the sign select and every iteration count from 0,
against the oracle (medians and counts exactly, trend to 1e-5)."""
import numpy as np
import pytest

import oracle
from paper_2604_06602_gb300 import synth
from tests.helpers import compare_diag

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chain", [1, 2, 3, 8, 9])
@pytest.mark.parametrize("W", [193, 361, 383])
def test_pairs(tmp_path, W, chain):
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    f = tmp_path / "force.txt"
    f.write_text("".join("%s|%d|%s|32|12|4|%d|128\n" % (torch.cuda.get_device_name(), W, r, chain)
                         for r in ("throughput", "latency")))
    umi.clear_tuning()
    try:
        umi.load_tuning(str(f))
        for n in (1, 2, W, 1500 + chain, 1501 + chain):
            x = synth.random_curve(W + chain + n, n, nan_frac=0.3, nan_runs=2, run_len=(1, W))
            x[n // 3:n // 3 + 60] = 1.0                     # zero scale inside a constant run
            for alpha, iters in ((2.0, 5), (6.0, 5), (0.2, 3), (2.0, 0), (2.0, 1)):
                p = umi.params(alpha=alpha, iters=iters, min_valid=40)
                got = umi.detrend_diag(torch.from_numpy(x).cuda(), W, p)
                torch.cuda.synchronize()
                compare_diag({k: v.cpu().numpy() for k, v in got.items()},
                             oracle.detrend(x, W, alpha=alpha, iters=iters, min_valid=40),
                             what="n=%d alpha=%g iters=%d" % (n, alpha, iters))
    finally:
        umi.clear_tuning()
