// umi_plan.cu -- the kernel planner and the tuned-plan table.
//
// A band is the set of windows of one length W (and scale mode) in a call.
// Its plan picks the kernel variant (G lanes per window, R slots per lane,
// register budget), the chain of positions each group walks, and the CTA
// size, by a rule fitted to measured plans on GB300; umi_autotune (timing
// runs in umi_api.cu) replaces the rule for a (W, regime) pair, and the table
// it fills can be saved to and loaded from a text file.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <fstream>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "umi_internal.h"

namespace umi {

bool legal_chain(int G, int chain)
{
    // The 32/G groups of a warp start `chain` positions apart in the tile, so
    // one slot row's loads read words g * chain + lane (g < 32/G, lane < G).
    // A chain of G * (odd number) positions keeps the groups on disjoint
    // banks; a chain of at most G makes the groups' words one contiguous run
    // of at most 32 (overlapping windows read the same words), so no two
    // distinct words share a bank either.
    if (chain < 1) return false;
    if (G >= 32 || chain <= G) return true;
    return chain % G == 0 && ((chain / G) & 1) == 1;
}

// Smallest legal chain of at least `target` positions.
int chain_at_least(int G, int64_t target)
{
    target = std::min<int64_t>(std::max<int64_t>(target, 1), 1 << 20);
    if (G >= 32) return (int)target;
    int64_t odd = (target + G - 1) / G;
    if ((odd & 1) == 0) ++odd;
    return (int)(G * odd);
}

int shortest_chain(int G) { return G >= 32 ? 1 : G; }
// Longest chain the planner uses: about 136 positions for groups of 8 or more
// lanes, about 33 for narrower groups (whose tile is already 32 windows wide).
int chain_cap(int G) { return chain_at_least(G, G >= 8 ? 136 : 33); }
static int default_threads(int G) { return G <= 2 ? 128 : 256; }

// Planning constants, measured on GB300 over window lengths 25 to 2161 and
// bands of 1e4 to 3e6 positions:
//  * the chain is sized so that about kWarpsPerSm warps per SM get a tile
//    (kWarpsPerSmNarrow for one- and two-lane groups in the latency regime);
//  * a band is in the latency regime when, even at the shortest chain of its
//    throughput variant, it has fewer than kLatencyItemsPerSm tiles per SM;
//  * below kRegisterRichBelow positions the variant with the larger register
//    budget wins (the tighter budget pays only once many warps share an SM);
//  * below kSmallCtaBelow positions 128-thread CTAs spread a band more evenly.
static const int kWarpsPerSm = 16;
static const int kWarpsPerSmNarrow = 8;
static const int kLatencyItemsPerSm = 32;
static const int64_t kRegisterRichBelow = 500000;
static const int64_t kSmallCtaBelow = 300000;

// Tuned plans, keyed by (window length, regime) (filled by umi_autotune /
// umi_load_tuning).  Every change bumps g_tune_epoch, which is part of the
// CUDA-graph cache key, so a cached graph never replays a plan that is no
// longer current.
static std::mutex g_tune_mu;
static std::map<std::pair<int, int>, Plan> g_tuned;
static std::atomic<uint64_t> g_tune_epoch{0};

static int smallest_capacity(int W)
{
    int n = 0;
    const Variant *t = variant_table(&n);
    int best = 1 << 30;
    for (int v = 0; v < n; ++v)
        if (t[v].G * t[v].R >= W) best = std::min(best, t[v].G * t[v].R);
    return best;
}

// Capacity S covers W and wastes at most a third of it (the smallest covering
// capacity always qualifies).
static bool tight_fit(const Variant &v, int W, int smallest)
{
    const int S = v.G * v.R;
    return S >= W && (S == smallest || 3 * S <= 4 * W);
}

// Variant for bands that fill the GPU: the smallest covering capacity; below
// kRegisterRichBelow positions, the tight fit with the largest register budget
// (lowest MINB), then the smallest capacity.
static int throughput_variant(int W, int64_t positions)
{
    int n = 0;
    const Variant *t = variant_table(&n);
    const int smallest = smallest_capacity(W);
    const bool rich = positions > 0 && positions < kRegisterRichBelow;
    int best = -1;
    for (int v = 0; v < n; ++v) {
        if (!tight_fit(t[v], W, smallest)) continue;
        if (best < 0) {
            best = v;
            continue;
        }
        const Variant &a = t[v], &b = t[best];
        const int Sa = a.G * a.R, Sb = b.G * b.R;
        if (rich ? (a.minb < b.minb || (a.minb == b.minb && Sa < Sb)) : Sa < Sb) best = v;
    }
    return best;
}

// Variant for bands too small to fill the GPU.  A group narrower than a warp
// needs a chain of at least G positions, so its tile is at least 32 windows
// and the band yields at most positions/32 tiles; a 32-lane group can run a
// chain of 1.  So when a 32-lane variant covers W within 2W (or is the
// smallest covering capacity), it is used -- a tight fit first, then the
// largest register budget, then the smallest capacity; otherwise the
// throughput variant stays.
static int latency_variant(int W, int64_t positions)
{
    int n = 0;
    const Variant *t = variant_table(&n);
    const int smallest = smallest_capacity(W);
    int best = -1;
    for (int v = 0; v < n; ++v) {
        const int S = t[v].G * t[v].R;
        if (t[v].G != 32 || S < W || (S != smallest && S > 2 * W)) continue;
        if (best < 0) {
            best = v;
            continue;
        }
        const Variant &a = t[v], &b = t[best];
        const bool ta = tight_fit(a, W, smallest), tb = tight_fit(b, W, smallest);
        if (ta != tb) {
            if (ta) best = v;
            continue;
        }
        if (a.minb != b.minb) {
            if (a.minb < b.minb) best = v;
            continue;
        }
        if (S < b.G * b.R) best = v;
    }
    return best >= 0 ? best : throughput_variant(W, positions);
}

int plan_regime(int W, int64_t positions)
{
    if (positions <= 0) return kRegimeThroughput;
    const int v = throughput_variant(W, positions);
    if (v < 0) return kRegimeThroughput;
    int n = 0;
    const Variant *t = variant_table(&n);
    const int G = t[v].G;
    const int64_t tile = (int64_t)(32 / G) * shortest_chain(G);
    const int64_t items = (positions + tile - 1) / tile;
    const int sms = std::max(1, device_info(current_device()).sms);
    return items < (int64_t)kLatencyItemsPerSm * sms ? kRegimeLatency : kRegimeThroughput;
}

// Chain for `positions` windows of a band in `regime`: about kWarpsPerSm
// warps per SM get a tile -- kWarpsPerSmNarrow for groups of one or two lanes
// in the latency regime, whose chain-start selects (a lane scans its whole
// window in every pass) cost more than the longer chains they save.  An untuned
// launch then fits its own (fit_launch).
static int chain_for(int G, int64_t positions, int regime)
{
    const int sms = std::max(1, device_info(current_device()).sms);
    const int target = (regime == kRegimeLatency && G <= 2) ? kWarpsPerSmNarrow : kWarpsPerSm;
    const int64_t warps = (int64_t)sms * target;
    const int64_t per_warp = (positions + warps - 1) / warps;  // windows per warp tile
    return chain_at_least(G, (per_warp * G + 31) / 32);       // 32/G groups share a tile
}

umi_status make_plan(int W, int64_t positions, Plan *plan)
{
    if (W < 1 || W > kMaxWindow || (W % 2) == 0)
        return fail(UMI_ERR_INVALID_ARG, "W must be odd and in [1, " + std::to_string(kMaxWindow) + "]");
    int n = 0;
    const Variant *t = variant_table(&n);
    const int regime = plan_regime(W, positions);
    Plan p;
    bool tuned = false;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tuned.find(std::make_pair(W, regime));
        if (it != g_tuned.end()) {
            p = it->second;
            p.tuned = tuned = true;
        }
    }
    if (!tuned) {
        const int v = regime == kRegimeLatency ? latency_variant(W, positions) : throughput_variant(W, positions);
        if (v < 0) return fail(UMI_ERR_INVALID_ARG, "no kernel variant for W=" + std::to_string(W));
        p.variant = v;
        p.G = t[v].G;
        p.R = t[v].R;
        p.threads = (positions > 0 && positions < kSmallCtaBelow) ? 128 : default_threads(p.G);
        p.chain = chain_cap(p.G);
    }
    // A band smaller than the chain was sized for gets a shorter chain, so
    // that its tiles still reach every SM: the rule's chain, or for a plan
    // tuned at a known band size the rule's chain times the ratio the tuner
    // preferred at that size (the tuned chain itself at the tuned size).
    if (positions > 0) {
        const int rule = std::min(chain_cap(p.G), chain_for(p.G, positions, regime));
        if (p.tuned_at <= 0) {
            p.chain = std::min(p.chain, rule);
        } else if (positions < p.tuned_at) {
            const int64_t at = std::min(chain_cap(p.G), chain_for(p.G, p.tuned_at, regime));
            p.chain = std::min(p.chain, chain_at_least(p.G, ((int64_t)rule * p.chain + at - 1) / at));
        }
    }
    p.regime = regime;
    *plan = p;
    return UMI_OK;
}

// A window's result depends on its variant, not on the chain it lies in, so a
// launch of an untuned plan fits the chain to its own curves.  With N steps
// (one window per group) for every resident warp, a chain of c steps costs
//     (tiles per warp) * (c + kStartSteps) + kTailTiles * (c + kStartSteps):
// each tile stages its samples and selects its first median, about three
// quarters of a step's work, and the launch ends with a partly idle tile;
// tiles are whole per curve (half a tile lost in each).  600 curves of 18,000
// samples at W = 361 (N = 1110): 5.35 ms at a chain of 136, 5.14 at 72, 5.09 at
// 56, 5.11 at 40; 32 of 118,000 at W = 2161 (N = 1552): 9.65 ms at 136, 9.53 at
// 48.  Bands of at most G steps per warp take the shortest chain that gives
// every resident warp one tile (chains up to G are bank-conflict free too):
// one curve of 18,000 samples at W = 721 43 us at a chain of 16, 33 at 8, 31 at
// 4, 35 at 2 (two tiles for some warps).  The MAD's one-window kernel of the paired
// variant takes the paired one's chain: 25.4 us at 6, 26.8 at its own 4.
//
// That cost knows no whole rounds, which decide where every warp gets a few tiles
// of equal length.  So in groups of 1 and 32 lanes, and of 2 for one curve, the
// result is held against the band's own chain and the chain of one tile per
// resident warp, by the steps of the busiest SM: one curve's tiles come in whole
// CTAs, as do a batch's that are all resident at once (its curves end unevenly,
// 20 %), and the last of them leave the SM partly filled.  Its warps' steps are
// faster then, nearly in proportion, but not in the variants of 8 warps per SM;
// and a start costs half a step in groups of one or two lanes.  A chain that is
// 6 % shorter by this count is taken: one curve of 300,000 samples at W = 4095
// 1.67 ms at 32, 1.48 at the band's 124 (two full rounds); one of 160,000 at W = 51
// 21.9 us at 1, 18.3 at 3; three of 118,000 at W = 17 31.7 at 1, 27.3 at 3.  Over
// 378 launches of 1 to 400 curves at W = 1 to 4095 the time is 2.5 % above the best
// chain's (geometric mean; without it 4.3 %, at the band's chain 9.9 %) and nowhere
// above what it is without it.  The other groups' steps do not follow the count
// (up to 5 % slower by it), nor do the paired windows', which are bound by latency;
// and curves that run in pieces (`split`) have tiles of all lengths: one of 1e6 in 90,000
// segments at W = 25 takes 0.84 ms by the first cost's chain, 1.25 by the count's.
void fit_launch(int64_t positions, int64_t n_curves, Plan *plan, bool split)
{
    static const double kStartSteps = 0.75, kTailTiles = 0.35;
    if (plan->tuned) return;
    int nv = 0;
    const Variant *t = variant_table(&nv);
    const int G = plan->G, groups = 32 / G;
    const bool pairs = pairs_windows(G, plan->R, 0);
    const int64_t warps =
        (int64_t)std::max(1, device_info(current_device()).sms) * 8 * (pairs ? 3 : t[plan->variant].minb);
    int64_t steps = (positions + warps * groups - 1) / (warps * groups);
    if (steps <= G) {
        if (pairs) steps += steps & 1;  // windows are worked on two at a time
        plan->chain = (int)std::max<int64_t>(1, steps);
        return;
    }
    const int cap = chain_cap(G), band_chain = plan->chain;
    double best = 1e300;
    for (int c = chain_at_least(G, 1); c <= cap; c = chain_at_least(G, c + 1)) {
        const double tiles = (double)positions / (groups * c) + 0.5 * (double)n_curves;
        const double cost = (std::max(1.0, tiles / (double)warps) + kTailTiles) * (c + kStartSteps);
        if (cost < best) {
            best = cost;
            plan->chain = c;
        }
        if (G >= 32 && c >= 16) c += 7;  // a coarser grid is enough there
    }
    if (split || pairs || (G > 2 && G < 32) || (G == 2 && n_curves > 1)) return;
    const int64_t cta_warps = plan->threads / 32, sms = warps / (8 * t[plan->variant].minb);
    const int64_t resident = 8 * t[plan->variant].minb / cta_warps;  // CTAs per SM
    auto busiest = [&](int c) {
        const int64_t windows = (int64_t)groups * c;
        const double tiles = n_curves == 1 ? (double)((positions + windows - 1) / windows)
                                           : (double)positions / (double)windows + 0.5 * (double)n_curves;
        double rounds = tiles / (double)warps + kTailTiles;
        if (n_curves == 1 || tiles <= (double)warps) {
            const int64_t ctas = ((int64_t)std::ceil(tiles) + cta_warps - 1) / cta_warps;
            const int64_t k = (ctas + sms - 1) / sms, rest = k % resident;
            const double idle = t[plan->variant].minb == 1 ? 1.0 : 0.1;  // pace of an empty SM
            rounds = (double)(k / resident);
            if (rest) rounds += idle + (1.0 - idle) * (double)rest / (double)resident;
            if (n_curves > 1) rounds *= 1.2;
        }
        return rounds * (c + (G <= 2 ? 0.5 : kStartSteps));
    };
    best = 0.94 * busiest(plan->chain);
    for (int c : {band_chain, chain_at_least(G, steps)}) {
        if (c > cap || busiest(c) >= best) continue;
        best = busiest(c);
        plan->chain = c;
    }
}

// The candidates umi_autotune times for a band: the variants that waste at
// most a third of W (the smallest covering capacity always qualifies) -- in
// the latency regime also the 32-lane variants within 2W --, two CTA sizes,
// and chains of about 8 to 136 positions plus a third, half, once, twice and
// three times the chain the rule gives for this band; in the latency regime
// groups narrower than a warp also try chains shorter than G (1, 2, 4, 6),
// which give a warp several windows in flight at once.
std::vector<Plan> autotune_candidates(int W, int64_t positions)
{
    const int regime = plan_regime(W, positions);
    int nv = 0;
    const Variant *t = variant_table(&nv);
    const int smallest = smallest_capacity(W);
    std::vector<Plan> out;
    for (int v = 0; v < nv; ++v) {
        const int S = t[v].G * t[v].R;
        const bool wide = regime == kRegimeLatency && t[v].G == 32 && S >= W && S <= 2 * W;
        if (!tight_fit(t[v], W, smallest) && !wide) continue;
        const int G = t[v].G;
        const int base = chain_for(G, positions, regime);
        std::vector<int> chains;
        for (int64_t target : {(int64_t)8, (int64_t)24, (int64_t)40, (int64_t)72, (int64_t)136,
                               (int64_t)base / 3, (int64_t)base / 2, (int64_t)base, 2 * (int64_t)base,
                               3 * (int64_t)base}) {
            const int c = chain_at_least(G, std::max<int64_t>(target, shortest_chain(G)));
            if (c <= chain_cap(G) + 2 * G && legal_chain(G, c) &&
                std::find(chains.begin(), chains.end(), c) == chains.end())
                chains.push_back(c);
        }
        if (regime == kRegimeLatency && G < 32)
            for (int c : {1, 2, 4, 6})
                if (c < G && std::find(chains.begin(), chains.end(), c) == chains.end()) chains.push_back(c);
        for (int threads : {128, 256}) {
            for (int c : chains) {
                Plan p;
                p.variant = v;
                p.G = G;
                p.R = t[v].R;
                p.threads = threads;
                p.chain = c;
                p.regime = regime;
                p.tuned_at = positions;
                out.push_back(p);
            }
        }
    }
    return out;
}

void store_tuned(int W, const Plan &p)
{
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned[std::make_pair(W, p.regime)] = p;
    ++g_tune_epoch;
}

uint64_t tune_epoch() { return g_tune_epoch.load(); }

void plan_out(const Plan &p, umi_plan *out)
{
    out->lanes = p.G;
    out->slots = p.R;
    out->chain = p.chain;
    out->threads = p.threads;
    out->variant = p.variant;
    out->latency = p.regime == kRegimeLatency ? 1 : 0;
}

}  // namespace umi

using namespace umi;

extern "C" {

umi_status umi_get_plan(int32_t W, int64_t positions, umi_plan *out)
{
    clear_error();
    if (!out) return fail(UMI_ERR_INVALID_ARG, "null plan");
    Plan p;
    umi_status st = make_plan(W, positions, &p);
    if (st != UMI_OK) return st;
    plan_out(p, out);
    return UMI_OK;
}

static const char *regime_name(int r) { return r == kRegimeLatency ? "latency" : "throughput"; }

umi_status umi_save_tuning(const char *path)
{
    clear_error();
    if (!path) return fail(UMI_ERR_INVALID_ARG, "null path");
    std::ofstream f(path);
    if (!f) return fail(UMI_ERR_INVALID_ARG, std::string("cannot write ") + path);
    const std::string gpu = device_info(current_device()).name;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    int nv = 0;
    const Variant *t = variant_table(&nv);
    f << "# umi tuning table: gpu|W|regime|G|R|MINB|chain|threads|positions\n";
    for (auto &kv : g_tuned)
        f << gpu << "|" << kv.first.first << "|" << regime_name(kv.first.second) << "|" << kv.second.G
          << "|" << kv.second.R << "|" << t[kv.second.variant].minb << "|" << kv.second.chain << "|"
          << kv.second.threads << "|" << kv.second.tuned_at << "\n";
    return UMI_OK;
}

umi_status umi_load_tuning(const char *path)
{
    clear_error();
    if (!path) return fail(UMI_ERR_INVALID_ARG, "null path");
    std::ifstream f(path);
    if (!f) return fail(UMI_ERR_INVALID_ARG, std::string("cannot read ") + path);
    const std::string gpu = device_info(current_device()).name;
    int nv = 0;
    const Variant *t = variant_table(&nv);
    std::string line;
    std::map<std::pair<int, int>, Plan> loaded;
    while (std::getline(f, line)) {
        if (line.empty() || line[0] == '#') continue;
        std::vector<std::string> parts;
        std::stringstream ss(line);
        std::string tok;
        while (std::getline(ss, tok, '|')) parts.push_back(tok);
        // Lines without a regime field are throughput plans; the band size
        // the plan was tuned at is optional (0: unknown).
        if (parts.size() == 7) parts.insert(parts.begin() + 2, "throughput");
        if (parts.size() == 8) parts.push_back("0");
        if (parts.size() != 9) return fail(UMI_ERR_INVALID_ARG, "bad tuning line: " + line);
        if (parts[0] != gpu) continue;
        int regime = -1;
        if (parts[2] == "throughput") regime = kRegimeThroughput;
        if (parts[2] == "latency") regime = kRegimeLatency;
        Plan p;
        const int W = std::atoi(parts[1].c_str());
        p.G = std::atoi(parts[3].c_str());
        p.R = std::atoi(parts[4].c_str());
        const int minb = std::atoi(parts[5].c_str());
        p.chain = std::atoi(parts[6].c_str());
        p.threads = std::atoi(parts[7].c_str());
        p.regime = regime;
        p.tuned_at = std::atoll(parts[8].c_str());
        for (int v = 0; v < nv; ++v)
            if (t[v].G == p.G && t[v].R == p.R && t[v].minb == minb) p.variant = v;
        if (regime < 0 || p.variant < 0 || W < 1 || (W % 2) == 0 || W > kMaxWindow || p.G * p.R < W ||
            !legal_chain(p.G, p.chain) || p.chain > (1 << 20) || p.threads < p.G || p.threads > 256 ||
            p.threads % 32 || p.tuned_at < 0)
            return fail(UMI_ERR_INVALID_ARG, "bad tuning line: " + line);
        loaded[std::make_pair(W, regime)] = p;
    }
    std::lock_guard<std::mutex> lk(g_tune_mu);
    for (auto &kv : loaded) g_tuned[kv.first] = kv.second;
    ++g_tune_epoch;
    return UMI_OK;
}

void umi_clear_tuning(void)
{
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned.clear();
    ++g_tune_epoch;
}

}  // extern "C"
