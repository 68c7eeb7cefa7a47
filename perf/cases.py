"""The work this library is used for, as measurable cases.

A case names a survey (its cadence sets the window), an entry point, the
number and lengths of the curves and the estimator's parameters; `prepare`
draws such light curves on the GPU, `run` detrends them once through the
public binding and `exact` evaluates the same estimator in 64 bits with plain
torch.  Lengths depend on the case alone, values on the seed alone.
"""
import math

import numpy as np
import torch

from paper_2604_06602_gb300 import umi

DAY = 86400.0

# Cadence in seconds, lengths of a curve (about a tenth of a sector up to a
# whole one, or a mission for the long cadence), and what the light curves
# hold: a one-day gap in mid-series, or three-day gaps every 90 days; spikes.
SURVEYS = {
    "tess20s": dict(cadence=20.0, n=(20000, 118000), gap="mid", spikes=0.01),
    "tess2min": dict(cadence=120.0, n=(4000, 20000), gap="mid", spikes=0.0),
    "ffi200s": dict(cadence=200.0, n=(2000, 12000), gap="mid", spikes=0.0),
    "ffi10min": dict(cadence=600.0, n=(1000, 4000), gap="mid", spikes=0.0),
    "kepler": dict(cadence=1764.0, n=(2000, 70000), gap="periodic", spikes=0.0),
}


def _case(name, call, survey, curves, n_min, n_max, window_d=0.5, alpha=2.0, c=5.0, mad=False):
    case = dict(call=call, survey=survey, curves=curves, n_min=n_min, n_max=n_max, window_d=window_d,
                alpha=alpha, c=c, mad=mad)
    return dict(case, name=name) if name else case


def listed():
    return [
        # A user looks at one star.  The smallest: one Kepler quarter (W = 25), launch and latency.
        _case("one-kepler-quarter", "detrend", "kepler", 1, 4400, 4400, alpha=3.0),
        # One TESS sector at 2 min (W = 361), the single-curve workload of the benchmark.
        _case("one-tess-2min", "detrend", "tess2min", 1, 18000, 18000),
        # The same star with a one-day window (W = 721), for long transits.
        _case("one-tess-day-window", "detrend", "tess2min", 1, 18000, 18000, window_d=1.0),
        # A thousand equal TESS curves: the benchmark's headline batch.
        _case("tess-2min-batch", "batched", "tess2min", 1000, 18000, 18000),
        # A survey chunk of TESS 2-min and Kepler curves of all lengths in one call (W = 361 and 25).
        _case("mixed-uneven", "batched", "mixed", 512, 0, 0),
        # 20-s cadence (W = 2161), spikes on 1 % of the samples.
        _case("tess-20s-batch", "batched", "tess20s", 32, 118000, 118000),
        # Full-frame images at 200 s (W = 217), whole sectors.
        _case("ffi-200s-batch", "batched", "ffi200s", 400, 11800, 11800),
        # Full-frame images at 10 min (W = 73), many short uneven curves.
        _case("ffi-10min-batch", "batched", "ffi10min", 1500, 1000, 3900),
        # The comparison estimator of the injection sweep: symmetric biweight, MAD scale.
        _case("mad-biweight", "batched", "tess2min", 200, 18000, 18000, alpha=1.0, mad=True),
        # The aggressive preset of the injection sweep.
        _case("aggressive", "batched", "tess2min", 300, 18000, 18000, alpha=10.0, c=2.5),
        # Kepler mission-long curves with gap handling (split at gaps, W = 25).
        _case("kepler-segmented", "segmented", "kepler", 256, 4000, 70000, alpha=3.0),
        # From pinned host buffers and back, copies inside: the end-to-end path.
        _case("tess-2min-host", "host", "tess2min", 500, 18000, 18000),
    ]


def draw(rng):
    call = rng.choice(["detrend", "batched", "batched", "batched", "segmented", "host"])
    survey = rng.choice(sorted(SURVEYS) + (["mixed"] if call != "detrend" else []))
    alpha, c, mad = rng.choice([(2.0, 5.0, False)] * 3 + [(3.0, 5.0, False), (10.0, 2.5, False), (1.0, 5.0, True)])
    if survey == "mixed":
        return _case(None, call, survey, int(round(math.exp(rng.uniform(math.log(8), math.log(600))))), 0, 0,
                     0.5, alpha, c, mad)
    s = SURVEYS[survey]
    window_d = rng.choice([0.5, round(math.exp(rng.uniform(math.log(0.3), math.log(0.94))), 3)])
    lo, hi = s["n"]
    n_max = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    n_min = n_max if call == "detrend" or rng.random() < 0.5 else rng.randint(max(lo // 2, 1), n_max)
    # No more window samples than the headline batch has (the MAD selects once more).
    most = 6e9 / (_window(s["cadence"], window_d) * n_max * (3 if mad else 1))
    curves = 1 if call == "detrend" else int(round(math.exp(rng.uniform(math.log(2), math.log(2000)))))
    return _case(None, call, survey, max(1, min(curves, int(most))), n_min, n_max, window_d, alpha, c, mad)


def _window(cadence_s, window_d):
    return int(round(window_d * DAY / cadence_s)) | 1


def _curves(case):
    """[(survey, n)] of the case: lengths spread evenly between its bounds."""
    out = []
    for b in range(case["curves"]):
        survey, lo, hi = case["survey"], case["n_min"], case["n_max"]
        if survey == "mixed":
            survey, lo, hi = ("tess2min", 5000, 20000) if b % 2 == 0 else ("kepler", 4000, 70000)
        out.append((survey, lo + int((hi - lo) * ((b * 0.6180339887498949 + 0.5) % 1.0))))
    return out


def _layout(case):
    curves = _curves(case)
    offsets = np.zeros(len(curves) + 1, np.int64)
    np.cumsum([n for _, n in curves], out=offsets[1:])
    W = np.array([_window(SURVEYS[s]["cadence"], case["window_d"]) for s, _ in curves], np.int32)
    return curves, offsets, W


def _flux(case, seed):
    """Flux around 1: sinusoids, red and white noise, flares, spikes, transits, NaN gaps."""
    curves, offsets, W = _layout(case)
    B, total = len(curves), int(offsets[-1])
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def u(lo, hi, log=False):
        r = torch.rand(B, generator=g, device=dev, dtype=torch.float64)
        return torch.exp(math.log(lo) + r * (math.log(hi) - math.log(lo))) if log else lo + r * (hi - lo)

    n = torch.tensor([n for _, n in curves], device=dev)
    cad = torch.tensor([SURVEYS[s]["cadence"] / DAY for s, _ in curves], device=dev, dtype=torch.float64)
    spikes = torch.tensor([SURVEYS[s]["spikes"] for s, _ in curves], device=dev, dtype=torch.float64)
    periodic = torch.tensor([SURVEYS[s]["gap"] == "periodic" for s, _ in curves], device=dev)
    who = torch.repeat_interleave(torch.arange(B, device=dev), n, output_size=total)
    k = torch.arange(total, device=dev) - torch.tensor(offsets[:-1], device=dev)[who]
    t = k * cad[who]
    span = n * cad
    sigma = u(2e-4, 5e-3, log=True)
    x = torch.ones(total, device=dev, dtype=torch.float64)
    for _ in range(3):
        x += u(2e-4, 2e-3)[who] * torch.sin(2 * math.pi * t / u(1.0, 10.0)[who] + u(0.0, 2 * math.pi)[who])
    # AR(1) red noise: the truncated geometric filter 1 + phi z + ... + phi^511 z^511.
    phi = 0.99
    red = torch.randn(total, generator=g, device=dev) * math.sqrt(1.0 - phi * phi)
    for j in range(9):
        d = 1 << j
        if d < total:
            red = torch.cat([red[:d], red[d:] + phi ** d * red[:-d]])
    x += sigma[who] * (0.5 * red + torch.randn(total, generator=g, device=dev))
    for _ in range(5):
        dt = t - (u(0.0, 1.0) * span)[who]
        x += torch.where(dt >= 0, 5e-3 * torch.exp(-dt.clamp(min=0) * (1440.0 / 10.0)), 0.0)
    if bool((spikes > 0).any()):
        r = torch.rand(total, generator=g, device=dev, dtype=torch.float64)
        x += torch.where(r < spikes[who], torch.where(r < 0.5 * spikes[who], 10.0, -10.0) * sigma[who], 0.0)
    period = u(1.0, 15.0)
    half = 0.5 * u(1.0, 8.0) / 24.0
    phase = torch.remainder(t - (u(0.0, 1.0) * period)[who] + 0.5 * period[who], period[who]) - 0.5 * period[who]
    x -= u(1e-4, 5e-2, log=True)[who] * ((half[who] - phase.abs()) / (0.2 * half[who])).clamp(0.0, 1.0)
    mid = (t - 0.5 * span[who]).abs() < 0.5
    every = torch.remainder(t + u(0.0, 85.0)[who], 90.0) >= 87.0
    x[torch.where(periodic[who], every, mid)] = float("nan")
    return x.to(torch.float32), offsets, W


def prepare(case, seed):
    flux, offsets, W = _flux(case, seed)
    p = umi.params(alpha=case["alpha"], c=case["c"],
                   scale_mode=umi.SCALE_MAD if case["mad"] else umi.SCALE_UPPER_RMS)
    state = dict(call=case["call"], flux=flux, offsets=offsets, W=W, p=p)
    if case["call"] == "host":  # a loader's pinned buffers, kept from batch to batch
        state["flux"] = flux.cpu().pin_memory()
        state["trend"] = torch.empty_like(state["flux"]).pin_memory()
        state["detr"] = torch.empty_like(state["flux"]).pin_memory()
    return state


def run(state):
    flux, offsets, W, p = state["flux"], state["offsets"], state["W"], state["p"]
    if state["call"] == "detrend":
        return umi.detrend(flux, int(W[0]), p)
    if state["call"] == "batched":
        return umi.detrend_batched(flux, offsets, W, p)
    if state["call"] == "segmented":
        return umi.detrend_segmented(flux, offsets, W, p)
    return umi.detrend_batched_host(flux, offsets, W, p, trend=state["trend"], detr=state["detr"])


def work(case):
    """Each sample is read once, its trend and detrended flux are written once.
    Per sample of a window: five iterations of nine operations (residual,
    scale, two for the sign select, 1 - u^2, clamp, square, two sums), five
    for the scale and four for one selection pass, one more for the MAD."""
    _, offsets, W = _layout(case)
    samples = sum(int(w) * int(n) for w, n in zip(W, np.diff(offsets)))
    return {"bytes": 12.0 * float(offsets[-1]), "flops": (58.0 if case["mad"] else 54.0) * samples}


def _bounds(case, flux, offsets, W):
    """First and one-past-last sample of the stretch each position's windows
    may reach into (its curve, or its segment of the curve), and the number of
    stretches; -1 where there is no output."""
    lo = np.full(flux.size, -1, np.int64)
    hi = np.full(flux.size, -1, np.int64)
    kept = 0
    for b, w in enumerate(W):
        a, e = int(offsets[b]), int(offsets[b + 1])
        if case["call"] != "segmented":
            lo[a:e], hi[a:e] = a, e
            continue
        at = a + np.flatnonzero(np.isfinite(flux[a:e]))
        if at.size == 0:
            continue
        cut = np.flatnonzero(np.diff(at) - 1 >= w) + 1
        for part in np.split(at, cut):
            if part.size >= w // 3:
                kept += 1
                lo[part[0]:part[-1] + 1], hi[part[0]:part[-1] + 1] = part[0], part[-1] + 1
    return lo, hi, kept


def exact(case, seed):
    if work(case)["flops"] > 54.0 * 9e9:
        return None  # too long in 64 bits
    flux, offsets, W = _flux(case, seed)
    dev = flux.device
    lo, hi, kept = _bounds(case, flux.cpu().numpy(), offsets, W)
    lo, hi = torch.from_numpy(lo).to(dev), torch.from_numpy(hi).to(dev)
    width = torch.repeat_interleave(torch.from_numpy(W.astype(np.int64)), torch.from_numpy(np.diff(offsets))).to(dev)
    trend = torch.full(flux.shape, float("nan"), dtype=torch.float64, device=dev)
    for w in sorted(set(W.tolist())):
        rows = torch.nonzero((width == w) & (lo >= 0) & torch.isfinite(flux)).reshape(-1)
        step = max(1, (1 << 26) // w)
        for r in range(0, rows.numel(), step):
            at = rows[r:r + step]
            trend[at] = _trend64(flux, at, lo[at], hi[at], w, case)
    detr = flux.double() / trend
    if case["call"] == "host":
        trend, detr = trend.cpu(), detr.cpu()
    return (trend, detr, kept) if case["call"] == "segmented" else (trend, detr)


def _trend64(flux, at, lo, hi, w, case):
    idx = at[:, None] + torch.arange(-(w // 2), w // 2 + 1, device=at.device)
    ok = (idx >= lo[:, None]) & (idx < hi[:, None])
    x = flux[idx.clamp_(0, flux.numel() - 1)]
    ok &= torch.isfinite(x)
    nv = ok.sum(1)
    rank = ((nv - 1) // 2)[:, None]
    inf = torch.tensor(float("inf"), device=at.device)
    m = torch.where(ok, x, inf).sort(1).values.gather(1, rank).double()
    y = torch.where(ok, x.double() - m, 0.0)
    if case["mad"]:
        s = torch.where(ok, y.abs(), inf.double()).sort(1).values.gather(1, rank)
    else:
        above = y > 0
        s = 0.6745 * torch.sqrt((y.clamp(min=0) ** 2).sum(1, keepdim=True) / above.sum(1, keepdim=True).clamp(min=1))
    cs = torch.where(s > 0, s * case["c"], 1.0)
    d = torch.zeros_like(m)
    for _ in range(5):
        v = (y - d) / cs
        v = torch.where(v < 0, case["alpha"] * v, v)
        wt = torch.where(ok & (v.abs() < 1), (1 - v * v) ** 2, 0.0)
        sw = wt.sum(1, keepdim=True)
        d = torch.where((s > 0) & (sw > 0), (wt * y).sum(1, keepdim=True) / sw.clamp(min=1e-300), d)
    mu = (m + d)[:, 0]
    return torch.where(nv >= w // 3, mu, float("nan"))
