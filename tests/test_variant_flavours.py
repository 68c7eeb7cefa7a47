"""Every kernel variant in each of its flavours, forced through a tuning file: both
forms of the sign select (alpha = 2 and 10) with both scales, with diagnostics
(detrend_diag) and without (detrend_batched), at the variant's capacity and
a little below it, on flux with gaps, spikes and ties, against the oracle; and
lengths at the edges of the tiles of a forced chain."""
import numpy as np
import pytest

import oracle
from paper_2604_06602_gb300 import synth
from tests.helpers import compare_detr, compare_diag, compare_trend
from tests.test_planner_host import variant_table

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def force(tmp_path):
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)

    def load(W, G, R, minb, chain, threads=128):
        f = tmp_path / "force.txt"
        # Tuned at one position: launches of any size take the chain as it stands.
        f.write_text("".join("%s|%d|%s|%d|%d|%d|%d|%d|1\n" % (torch.cuda.get_device_name(), W, r, G, R, minb, chain,
                                                            threads) for r in ("throughput", "latency")))
        umi.clear_tuning()
        umi.load_tuning(str(f))
        return umi

    yield load
    umi.clear_tuning()


@pytest.mark.parametrize("v", variant_table(), ids=lambda v: "%d-%d-%d" % v)
def test_flavours(force, v):
    G, R, minb = v
    S = G * R
    for W in sorted({min(4095, S - 1 + S % 2), min(4095, int(0.98 * S) | 1)}):
        umi = force(W, G, R, minb, 5 if G >= 32 else G)
        n = min(2 * W + 100, W + 400)
        x = synth.random_curve(7 * S + W, n, nan_frac=0.03, nan_runs=2, run_len=(1, max(2, W // 3)), quantum=1e-5)
        x[n // 5::17] += np.float32(0.02)
        xd = torch.from_numpy(np.concatenate([x, x[::-1]])).cuda()
        off = np.array([0, n, 2 * n], np.int64)
        for alpha in (2.0, 10.0):
            for mode in (umi.SCALE_UPPER_RMS, umi.SCALE_MAD):
                p = umi.params(alpha=alpha, min_valid=3, scale_mode=mode)
                what = "W=%d alpha=%g mode=%d" % (W, alpha, mode)
                ref = oracle.detrend(x, W, alpha=alpha, min_valid=3, scale_mode=mode)
                got = umi.detrend_diag(xd[:n], W, p)
                tr, de = umi.detrend_batched(xd, off, np.full(2, W, np.int32), p)
                torch.cuda.synchronize()
                compare_diag({k: t.cpu().numpy() for k, t in got.items()}, ref, what=what)
                compare_trend(tr[:n].cpu().numpy(), ref["trend"], what=what + " batched")
                compare_detr(de[:n].cpu().numpy(), ref["detr"], what=what + " batched")


@pytest.mark.parametrize("W,v,chain", [(3, (1, 8, 4), 5), (25, (1, 26, 4), 3), (25, (1, 32, 3), 1),
                                       (73, (2, 38, 2), 6), (217, (4, 56, 2), 12), (361, (8, 46, 2), 24),
                                       (361, (32, 12, 4), 1), (361, (32, 12, 4), 2), (361, (32, 12, 4), 7),
                                       (193, (32, 12, 4), 8), (721, (16, 48, 2), 16), (2161, (32, 68, 2), 9)])
def test_lengths_at_tile_edges(force, W, v, chain):
    umi = force(W, *v, chain)
    assert umi.get_plan(W, 3)["chain"] == chain
    T = 32 // v[0] * chain
    for n in sorted({max(1, k * T + d) for k in (1, 2, 3) for d in (-1, 0, 1)}):
        x = synth.random_curve(50 + n, n, nan_runs=1, run_len=(1, max(2, W // 4)))
        for alpha in (2.0, 6.0):
            ref = oracle.detrend(x, W, alpha=alpha, min_valid=1)
            got = umi.detrend_diag(torch.from_numpy(x).cuda(), W, umi.params(alpha=alpha, min_valid=1))
            torch.cuda.synchronize()
            compare_diag({k: t.cpu().numpy() for k, t in got.items()}, ref, what="W=%d n=%d alpha=%g" % (W, n, alpha))
