"""The kernel's rank select (the chain-start median and the MAD) and its rank walk
along a chain on value distributions they can go wrong on, against the oracle: medians, valid
counts and above-median counts exactly.  The MAD is an order statistic of
fl(|x - m|), each one rounding of the exact |x - m| and monotone in it, so it
is the rounding of the exact MAD: one unit of FP32 (relative 2^-23, or one
subnormal step) bounds the difference."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def curves(n, W):
    rng = np.random.default_rng(31 * W + n)
    noise = rng.normal(0.0, 1e-3, n)
    out = {
        "two_levels": np.where(rng.random(n) < 0.5, 0.5, 1.5) + noise,
        "step": np.where(np.arange(n) % (2 * W) < W, 1.0, 1.02) + noise,
        "outliers": 1.0 + noise + np.where(rng.random(n) < 0.02, rng.choice([-1e6, 1e6], n), 0.0),
        "signed_zeros": rng.choice(np.array([-0.0, 0.0, -0.0, 0.0, 1e-3, -1e-3, 2.0]), n),
        "subnormal": rng.integers(-40, 41, n) * 2.0 ** -149,
        "powers": np.exp2(rng.integers(-59, 59, n).astype(float)) * rng.choice([-1.0, 1.0], n),
        "negative": -1.0 + noise,
        "around_zero": noise,
        # Median and neighbours on both sides of zero (the rank walk's two forms).
        "sign_edge": rng.choice([-1.0, 1.0], n) * rng.uniform(0.5, 2.0, n),
        "mostly_positive": np.abs(noise) - np.where(rng.random(n) < 0.45, 3e-3, 0.0),
        "levels": 1.0 + 1e-3 * rng.integers(0, 4, n),
        "sparse": np.where(rng.random(n) < 2.5 / W, 1.0 + noise, np.nan),
        "gaps": 1.0 + noise,
    }
    out["gaps"][np.arange(n) % (3 * W) < W + 2] = np.nan
    out["signed_zeros"][rng.random(n) < 0.1] = np.nan
    return {k: v.astype(np.float32) for k, v in out.items()}


@pytest.mark.parametrize("mad", [False, True])
@pytest.mark.parametrize("W", [1, 3, 25, 51, 73, 151, 217, 361, 543, 721, 2161, 3071])
def test_rank_select_is_exact(W, mad):
    from paper_2604_06602_gb300 import umi
    umi.load(build_if_missing=True)
    p = umi.params(min_valid=0, scale_mode=umi.SCALE_MAD if mad else umi.SCALE_UPPER_RMS)
    n = min(4 * W + 203, W + 700)
    for name, x in curves(n, W).items():
        out = umi.detrend_diag(torch.from_numpy(x).cuda(), W, p)
        torch.cuda.synchronize()
        got = {k: v.cpu().numpy() for k, v in out.items()}
        ref = oracle.detrend(x, W, min_valid=0, scale_mode=oracle.SCALE_MAD if mad else oracle.SCALE_UPPER_RMS)
        what = "%s W=%d" % (name, W)
        np.testing.assert_array_equal(got["nvalid"], ref["nvalid"], err_msg=what)
        np.testing.assert_array_equal(got["nplus"], ref["nplus"], err_msg=what)
        np.testing.assert_array_equal(got["median"].astype(np.float64), ref["median"], err_msg=what)
        if mad:
            ok = np.isfinite(ref["scale"])
            np.testing.assert_array_equal(np.isfinite(got["scale"]), ok, err_msg=what)
            np.testing.assert_allclose(got["scale"][ok], ref["scale"][ok], rtol=2.0 ** -23, atol=2.0 ** -149,
                                       err_msg=what)
