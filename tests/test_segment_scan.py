"""The device scan of the gap split at its word and chunk edges: curves that start
at any offset of the validity mask, gaps across the 64-sample words and across
the 65,536-sample chunks, splitting runs of 1, 63, 64, 65 and 200 samples, and
segments at the minimum's edge, against the oracle's segments."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def curve(rng, n):
    x = (1.0 + rng.normal(0.0, 1e-3, n)).astype(np.float32)
    for gap in (1, 2, 62, 63, 64, 65, 66, 199, 200, 201):
        for s in rng.integers(-gap, n, 6):
            x[max(0, s):max(0, s + gap)] = np.nan
    for edge in range(65536, n, 65536):              # gaps that end at, span and start at a chunk's edge
        a, b = [(edge - 70, edge), (edge - 130, edge + 90), (edge, edge + 64)][rng.integers(3)]
        x[a:b] = np.nan
    return x


@pytest.mark.parametrize("gap_min,min_seg", [(1, 0), (1, 30), (63, -1), (64, 64), (65, -1), (200, 500), (0, -1)])
def test_scan_edges(gap_min, min_seg):
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    rng = np.random.default_rng(1000 + 7 * gap_min + min_seg)
    W = 5
    lens = [1, 63, 64, 65, 127, 2000, 65535, 65536, 65537, 140001, 3]
    xs = [curve(rng, n) for n in lens]
    xs[1][:] = np.nan
    xs[5][::2] = np.nan
    flux = np.concatenate(xs)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tr, _, kept = umi.detrend_segmented(torch.from_numpy(flux).cuda(), off, np.full(len(lens), W, np.int32),
                                        gap_min=gap_min, min_seg=min_seg)
    torch.cuda.synchronize()
    tr = tr.cpu().numpy()
    n_ref = 0
    for k, x in enumerate(xs):
        rt, _, rk = oracle.detrend_segmented(x, W, gap_min=gap_min, min_seg=min_seg)
        n_ref += rk
        got = tr[off[k]:off[k + 1]]
        np.testing.assert_array_equal(np.isnan(got), np.isnan(rt), err_msg="curve %d" % k)
        ok = ~np.isnan(rt)
        np.testing.assert_allclose(got[ok], rt[ok], rtol=1e-5, err_msg="curve %d" % k)
    assert kept == n_ref
