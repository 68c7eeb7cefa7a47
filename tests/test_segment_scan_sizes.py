"""The gap split's scan in each of its CTA sizes (the longest curve of a call picks
it): curves that end at, before and after a chunk's edge and at the size where the
next CTA takes over, gaps and segments across chunks, words with many
segment starts; and curves too short to keep a segment beside ones that do.
Against the oracle's segments, and bit for bit against the plain call where no
curve splits."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = {1: [1, 2, 2047, 2048, 2049, 3000, 4095, 4096],
         8: [5, 4097, 16383, 16384, 16385, 20000, 32767, 32768],
         32: [7, 2048, 32769, 65536, 65537]}


def curve(rng, n, dense):
    x = (1.0 + rng.normal(0.0, 1e-3, n)).astype(np.float32)
    for gap in (1, 2, 63, 64, 65, 130, 2100):
        for s in rng.integers(-gap, n, 3):
            x[max(0, s):max(0, s + gap)] = np.nan
    for edge in range(2048, n, 2048):
        a, b = [(edge - 70, edge), (edge - 3, edge + 90), (edge, edge + 64), (edge, edge)][rng.integers(4)]
        x[a:b] = np.nan
    if dense:
        x[rng.random(n) < 0.4] = np.nan
    return x


@pytest.mark.parametrize("gap_min,min_seg", [(1, 1), (2, 0), (64, -1), (100, 2500)])
@pytest.mark.parametrize("warps", sorted(EDGES))
@pytest.mark.parametrize("dense", [False, True])
def test_scan_of_each_size(warps, gap_min, min_seg, dense):
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    rng = np.random.default_rng(100 * warps + gap_min + dense)
    lens = EDGES[warps]
    xs = [curve(rng, n, dense) for n in lens]
    flux = np.concatenate(xs)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    W = np.array([(5, 361)[k % 2] for k in range(len(lens))], np.int32)
    tr, de, kept = umi.detrend_segmented(torch.from_numpy(flux).cuda(), off, W, gap_min=gap_min, min_seg=min_seg)
    torch.cuda.synchronize()
    tr, de = tr.cpu().numpy(), de.cpu().numpy()
    n_ref = 0
    for k, x in enumerate(xs):
        rt, rd, rk = oracle.detrend_segmented(x, int(W[k]), gap_min=gap_min, min_seg=min_seg)
        n_ref += rk
        for got, ref in ((tr[off[k]:off[k + 1]], rt), (de[off[k]:off[k + 1]], rd)):
            np.testing.assert_array_equal(np.isnan(got), np.isnan(ref), err_msg="curve %d" % k)
            ok = ~np.isnan(ref)
            np.testing.assert_allclose(got[ok], ref[ok], rtol=1e-5, err_msg="curve %d" % k)
    assert kept == n_ref


def test_curves_too_short_for_a_segment():
    """They are planned with the others (same bits as the plain call) and give NaN; a call of nothing else
    keeps no segment."""
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    rng = np.random.default_rng(9)
    lens = [119, 4000, 3, 120, 60000, 118, 121]
    x = torch.from_numpy((1.0 + rng.normal(0.0, 1e-3, sum(lens))).astype(np.float32)).cuda()
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    W = np.full(len(lens), 361, np.int32)
    tr, de, kept = umi.detrend_segmented(x, off, W)
    pt, pd = umi.detrend_batched(x, off, W)
    assert kept == 4
    for k, n in enumerate(lens):
        for got, ref in ((tr, pt), (de, pd)):
            got, ref = got[off[k]:off[k + 1]], ref[off[k]:off[k + 1]]
            if n < 120:
                assert torch.isnan(got).all()
            else:
                assert torch.equal(got.view(torch.int32), ref.view(torch.int32))
    tr, de, kept = umi.detrend_segmented(x, off, W, min_seg=60001)
    assert kept == 0 and torch.isnan(tr).all() and torch.isnan(de).all()
