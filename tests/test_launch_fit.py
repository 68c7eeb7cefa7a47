"""A launch fits its chain to its curves.  Results must depend neither on it nor on
the CTA size: whatever the launch chose equals, bit for bit, the same variant forced
through a tuning file with other chains and CTA sizes; and the curve that owns
a work item is found for batches on both sides of each round of the search
(32 and 1024 curves), with lengths that leave partial tiles."""
import numpy as np
import pytest

from paper_2604_06602_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def umi():
    from paper_2604_06602_gb300 import umi as u
    u.load(build_if_missing=True)
    return u


def minb_of(index):
    from tests.test_planner_host import variant_table
    return variant_table()[index][2]


@pytest.mark.parametrize("W", [3, 25, 49, 73, 145, 217, 361, 433, 721, 1621, 2161])
@pytest.mark.parametrize("curves,n", [(1, 37), (1, 4400), (1, 18000), (31, 130), (33, 1000), (1025, 61), (40, 9001)])
def test_results_do_not_depend_on_the_launch_shape(umi, tmp_path, W, curves, n):
    rng = np.random.default_rng(W + curves)
    lens = np.maximum(1, n - rng.integers(0, 30, curves))
    x = synth.random_curve(60 + W, int(lens.sum()), nan_frac=0.02, nan_runs=3, run_len=(1, 200))
    flux = torch.from_numpy(x).cuda()
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    Wv = np.full(curves, W, np.int32)
    umi.clear_tuning()
    plan = umi.get_plan(W, int(lens.sum()))
    t0, d0 = umi.detrend_batched(flux, off, Wv)
    G = plan["lanes"]
    try:
        for chain, threads in ((1, 256), (G * 3 if G < 32 else 7, 128), (G * 5 if G < 32 else 60, 64)):
            f = tmp_path / "force.txt"
            f.write_text("".join("%s|%d|%s|%d|%d|%d|%d|%d\n" % (torch.cuda.get_device_name(), W, r, G, plan["slots"],
                                                                minb_of(plan["variant"]), chain, threads)
                                 for r in ("throughput", "latency")))
            umi.load_tuning(str(f))
            t1, d1 = umi.detrend_batched(flux, off, Wv)
            assert torch.equal(t0.view(torch.int32), t1.view(torch.int32)), (chain, threads)
            assert torch.equal(d0.view(torch.int32), d1.view(torch.int32)), (chain, threads)
    finally:
        umi.clear_tuning()
