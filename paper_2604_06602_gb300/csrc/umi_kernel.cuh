// umi_kernel.cuh -- sm_103a kernel for the UMI sliding-window robust trend.
//
// Method (paper Section 2): per output position, over the W-sample window
// with missing samples dropped: Phase 1 exact median (Section 2.1), Phase 2
// upper-RMS scale s = 0.6745 sqrt(mean_{x > m} (x - m)^2) (Eq. 1), Phase 3
// `iters` asymmetric bisquare reweighting steps (Eqs. 2-4), trend = mu,
// detrended flux = x / mu.
//
// GPU design (not the paper's one-thread-per-window kernel, Section 2.6):
//  * A warp owns a tile of T consecutive positions of one curve and stages the
//    T + S - 1 samples its windows touch into its slice of shared memory once,
//    with 4-byte cp.async copies; missing samples (non-finite, or outside the
//    curve) become kGap.
//  * A "group" of G lanes (G = 1..32, a power of two) evaluates one window at a
//    time, each lane holding R window slots in registers (S = G*R >= W slots;
//    slots past W hold kGap).  The 32/G groups of a warp run in lock step on
//    neighbouring chains; every block that shuffles is entered warp-uniformly.
//  * Each group walks a chain of P consecutive positions.  At the chain start
//    (or after an empty window) the median comes from an exact rank select
//    over the registers.  Afterwards the group keeps the
//    counts L = #{x < m}, E = #{x == m}, G+ = #{x > m} of the current window
//    and updates them in O(1) per step from the sample that leaves and the one
//    that enters.  One step moves the median's rank by at most one, so the new
//    median is m itself, the largest sample below m, or the smallest above m;
//    the last two take one pass over the registers.  Every median is the exact
//    order statistic of rank floor((n_valid - 1)/2).
//  * Eq. 1 is one pass over the registers, G+ comes from the counts.
//  * Phase 3 keeps y = x - m in registers, in pairs for the packed FP32x2
//    instructions, and runs the fixed number of steps on mu = m + delta: per
//    slot u_eff^2 = t (t + rho |t|) with t = sigma (y - delta) (for
//    1/4 <= alpha <= 4; otherwise u_eff = min(y kp - delta kp, y kn - delta
//    kn) with kp = 1/(c s), kn = alpha/(c s): Eq. 2 without a branch either
//    way), z = sat(1 - u_eff^2), w = z^2 (Eq. 3), and delta = sum(w y)/sum(w)
//    (Eq. 4 about m).  A kGap slot has u_eff^2 >= 1 (or it overflows, or is
//    NaN), so sat() makes its weight exactly 0 without a mask.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace umi {

// Missing-sample marker inside the tile.  Finite, below every admissible
// sample (|x| < 2^60), and so far below that its standardised residual never
// reaches the bisquare support.
constexpr float kGap = -0x1p100f;
constexpr float kGapLimit = -0x1p99f;  // x > kGapLimit  <=>  a real sample
constexpr float kScaleFactor = 0.6745f;  // Section 2.2, as printed

struct Curve {
    const float *flux;
    float *trend;
    float *detr;
    int64_t n;
    int32_t W;
    int32_t min_valid;  // resolved, >= 0
    float alpha;
    float c;
    int32_t iters;
    int32_t scale_mode;  // 0: upper-RMS scale (Eq. 1); 1: MAD
};

struct Diag {
    float *median;
    int32_t *nvalid;
    int32_t *nplus;
    float *scale;
};

// A work item is one tile of T = (32/G)*P positions of one curve.  Items are
// numbered through the launch's curves: curve c owns the items first_tile[c]
// .. first_tile[c + 1] - 1 (the last one up to n_items - 1).
struct LaunchArgs {
    const Curve *curves;  // device curve table of the launch, or nullptr to use `single`
    Curve single;
    const int32_t *first_tile;  // [n_curves], ascending from 0 (unused with `single`)
    int32_t n_items;
    int32_t chain;        // P: consecutive positions per group
    uint32_t *queue;      // persistent work counter (0 between launches), or
                          // nullptr: one item per warp
    Diag diag;
    int32_t n_curves;     // entries of `curves`
    uint32_t *check;      // checked builds: flag word of failed index checks
};

// Index checks of the checked build (compiled with UMI_CHECKED).  A failed
// check sets its bit in LaunchArgs::check and the access is skipped (a read
// gives kGap, a write is dropped), so a bad index is reported, never
// performed.  Normal builds compile none of it.
enum : uint32_t {
    kCheckSmemSize = 1u << 0,    // the warps' tile slices exceed the launch's dynamic smem
    kCheckTileRead = 1u << 1,    // window, slide or centre read outside the warp's tile
    kCheckCurveIndex = 1u << 2,  // work item found no curve, or one outside the table
    kCheckItemTile = 1u << 3,    // work item's tile starts past its curve's end
};

// Read-only view of a warp's tile: a bare pointer in normal builds, a
// bounds-checked reader in checked builds.
struct TileRef {
    const float *p;
#ifdef UMI_CHECKED
    int len;
    uint32_t *check;
    __device__ __forceinline__ float operator[](int i) const
    {
        if (i < 0 || i >= len) {
            if (check) atomicOr(check, kCheckTileRead);
            return kGap;
        }
        return p[i];
    }
#else
    __device__ __forceinline__ float operator[](int i) const { return p[i]; }
#endif
};

// ---- group-wide reductions over G aligned lanes --------------------------
template <int G>
__device__ __forceinline__ float group_sum(float v)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int G>
__device__ __forceinline__ int group_sum_int(int v)
{
    if constexpr (G == 32) {
        return (int)__reduce_add_sync(0xffffffffu, (unsigned)v);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
}

template <int G>
__device__ __forceinline__ float group_max(float v)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int G>
__device__ __forceinline__ unsigned group_umin(unsigned v)
{
    if constexpr (G == 32) {
        return __reduce_min_sync(0xffffffffu, v);
    } else {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    }
}

// d = clamp(a*b + c, 0, 1), NaN -> 0, as one saturating FMA.
__device__ __forceinline__ float fma_sat(float a, float b, float c)
{
    float d;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// 1.0f when a >= b, else 0.0f (one compare, result as a float).
__device__ __forceinline__ float ge_flag(float a, float b)
{
    float d;
    asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// 1.0f when a <= b, else 0.0f (also 0.0f when either is NaN).
__device__ __forceinline__ float le_flag(float a, float b)
{
    float d;
    asm("set.le.f32.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// 1.0f when a == b, else 0.0f.
__device__ __forceinline__ float eq_flag(float a, float b)
{
    float d;
    asm("set.eq.f32.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// 4-byte asynchronous copy from global to shared memory (cp.async): the copy
// is issued without waiting for it, so a lane's staging loads are all in
// flight at once; cp_async_wait_all waits for the calling thread's copies.
__device__ __forceinline__ void cp_async4(float *smem_dst, const float *gmem_src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Order-preserving map from non-NaN floats to unsigned keys (-0 sorts just
// below +0; the counts that follow compare floats, where they are equal).
__device__ __forceinline__ unsigned float_key(float f)
{
    unsigned b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float key_float(unsigned k)
{
    unsigned b = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(b);
}

// Key of a sample for the selects: the order-preserving key, or for magnitudes
// (ABS) the bit pattern, whose unsigned order is their order.
template <bool ABS>
__device__ __forceinline__ unsigned sel_key(float f)
{
    return ABS ? __float_as_uint(f) : float_key(f);
}

template <bool ABS>
__device__ __forceinline__ float sel_float(unsigned k)
{
    return ABS ? __uint_as_float(k) : key_float(k);
}

// Exact selection over the S slots of each group that `need`s it: the sample v
// (|v| with ABS) of rank `target`, i.e. #{< v} <= target < #{<= v}.  The key
// interval [lo, hi] holds it; clo slots lie below lo and chi at or below hi
// (float order: -0 and +0 are equal, and an end that is a zero takes in both).
// *le returns #{<= v}, where it is known: *below says that instead
// #{< v} = target.
//
// Each pass counts the slots at or below a pivot.  Bisecting the keys took
// about 17 passes for flux around 1.0 (18 with a transit in the window); the
// pivot is where the rank would lie if the samples between the ends were
// evenly spread, and the search stops as soon as the rank gap is known:
// clo = target (the answer is the smallest sample above) or chi = target + 1
// (the largest one below), 5 to 7 passes and one that picks the sample.  Every
// eighth pass moves the ends onto samples, which ends the search when ties
// fill the interval, and from the sixth pass on every second pivot bisects,
// so no input takes more than twice the key width.  One TESS curve (a select
// every 8 windows) 26.2 -> 25.1 us.  `q`, `dq`: first pivot
// and the spacing of one rank there (dq > 0), for the first three pivots.
// BITS: positive samples may be picked by their bit patterns.
template <int G, int R, bool ABS, bool BITS = true>
__device__ __forceinline__ float select_rank(const float2 (&x)[R / 2], bool need, unsigned lo, unsigned hi,
                                             int clo, int chi, int target, float q, float dq, int *le,
                                             bool *below)
{
    constexpr int kTighten = ABS ? 3 : 7;  // the magnitudes' first upper end is no sample
    float v;
    for (int p = 0;; ++p) {
        const bool more = __any_sync(0xffffffffu, need && lo < hi && clo != target && chi != target + 1);
        if (!more && (ABS || (BITS && __all_sync(0xffffffffu, !need || lo > 0x80000000u)))) {
            // Magnitudes, and samples above zero, are ordered as their bits
            // are: the answer is the pattern nearest to lo from above, or to hi
            // from below, both a smallest unsigned difference (the other
            // patterns, negative samples among them, are further away or
            // wrap).
            const bool up = clo == target;
            const unsigned lob = lo & 0x7fffffffu, hib = hi & 0x7fffffffu;
            const unsigned flip = up ? 0u : 0xffffffffu, add = up ? 0u - lob : hib + 1u;
            unsigned r0 = 0xffffffffu, r1 = 0xffffffffu;
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                const unsigned a = __float_as_uint(x[k].x), b = __float_as_uint(x[k].y);
                r0 = __viaddmin_u32((ABS ? a & 0x7fffffffu : a) ^ flip, add, r0);
                r1 = __viaddmin_u32((ABS ? b & 0x7fffffffu : b) ^ flip, add, r1);
            }
            const unsigned r = group_umin<G>(min(r0, r1));
            *below = up;
            *le = chi;
            return __uint_as_float(up ? lob + r : hib - r);
        }
        if (!more || (p & 7) == kTighten) {
            // Smallest sample above lo - 1 and largest at or below hi.
            const float lof = ABS ? (lo ? sel_float<ABS>(lo - 1) : -1.f) : sel_float<ABS>(lo - 1);
            const float hif = sel_float<ABS>(hi);
            float mn = INFINITY, mx = -INFINITY;
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                const float a = ABS ? fabsf(x[k].x) : x[k].x, b = ABS ? fabsf(x[k].y) : x[k].y;
                mn = fminf(mn, fminf(a > lof ? a : INFINITY, b > lof ? b : INFINITY));
                mx = fmaxf(mx, fmaxf(a <= hif ? a : -INFINITY, b <= hif ? b : -INFINITY));
            }
            mn = -group_max<G>(-mn);
            mx = group_max<G>(mx);
            if (!more) {
                *below = clo == target;
                *le = chi;
                v = clo == target ? mn : mx;
                break;
            }
            if (need) {
                lo = ABS ? __float_as_uint(mn) : (mn == 0.f ? 0x7fffffffu : float_key(mn));
                hi = ABS ? __float_as_uint(mx) : (mx == 0.f ? 0x80000000u : float_key(mx));
            }
        }
        const float fl = sel_float<ABS>(lo), fh = sel_float<ABS>(hi);
        float piv = fl + (fh - fl) * __fdividef(target + 0.5f - clo, (float)max(chi - clo, 1));
        if (dq > 0.f && p < 3 && q > fl && q < fh) piv = q;
        unsigned mid = min(max(sel_key<ABS>(piv), lo), max(hi, 1u) - 1u);
        if (p >= 6 && (p & 1)) mid = lo + ((hi - lo) >> 1);
        const float midf = sel_float<ABS>(mid);
        int c = 0;
        if constexpr (R >= 32) {
            // 0/1 float flags summed with FADD2 (exact: at most R < 2^24),
            // so half of a long pass runs on the FMA pipe.
            // Two accumulators (even and odd pairs) halve the
            // dependent chain; the count is exact in any order.
            float2 cf0 = make_float2(0.f, 0.f), cf1 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                const float2 f = make_float2(le_flag(ABS ? fabsf(x[k].x) : x[k].x, midf),
                                             le_flag(ABS ? fabsf(x[k].y) : x[k].y, midf));
                if (k & 1) cf1 = __fadd2_rn(cf1, f);
                else cf0 = __fadd2_rn(cf0, f);
            }
            c = (int)((cf0.x + cf0.y) + (cf1.x + cf1.y));
        } else {
#pragma unroll
            for (int k = 0; k < R / 2; ++k)
                c += (((ABS ? fabsf(x[k].x) : x[k].x) <= midf) ? 1 : 0) +
                     (((ABS ? fabsf(x[k].y) : x[k].y) <= midf) ? 1 : 0);
        }
        c = group_sum_int<G>(c);
        if (lo < hi && clo != target && chi != target + 1) {
            if (c > target) {
                hi = mid;
                chi = c;
            } else {
                lo = mid + 1;
                clo = c;
            }
        }
        q = midf + (target + 0.5f - c) * dq;
    }
    return v;
}

// a b + c per component, as one packed instruction or two scalar ones (the
// same values either way).
template <bool SCALAR>
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    return SCALAR ? make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)) : __ffma2_rn(a, b, c);
}

// Which of the iteration's FMAs are scalar pairs.  The FMA pipe takes about two
// cycles for a packed instruction and about one for a scalar one, alone or
// between packed ones (16 warps per SM: FFMA2 2.18, two FFMA 2.42, FFMA2 and FFMA
// 3.17, FFMA2 and two FFMA 4.27), so the mixes cost nearly the same there, but
// some are scheduled better.  Each lane split has the mix that those of its variants
// that were measured like best of 32; the others, (2,44), (4,38), (8,40), (8,48),
// (8,56), (16,40), (32,56) and (32,92) on among them, take the mix of the nearest
// measured one unmeasured (kernel times, all packed against it: W = 25
// (1,26) 0.576 -> 0.569 ms, W = 49 (1,52) 0.566 -> 0.550, W = 73 (2,38) 0.647 ->
// 0.633, W = 97 (2,52) 0.662 -> 0.647, W = 217 (4,56) 1.342 -> 1.329, W = 361
// (8,46) 2.595 -> 2.515, W = 541 (8,68) 1.839 -> 1.829, W = 721 (16,48) 1.807 ->
// 1.795, W = 1441 (32,48) 1.916 -> 1.894, W = 2161 (32,68) 9.41 -> 9.39; (4,46),
// (16,56) and (16,68) have none that is better).  The min form's second
// residual is scalar everywhere (alpha = 10: W = 361 2.851 -> 2.759 ms, W = 73
// 0.713 -> 0.684, W = 2161 5.444 -> 5.404).
struct IterationForm {
    bool t;    // t = sigma (y - delta)
    bool v;    // t + rho |t|
    bool swy;  // sum w y
};
__host__ __device__ constexpr IterationForm iteration_form(int G, int R)
{
    return G == 1    ? IterationForm{true, false, true}
           : G == 2  ? IterationForm{R <= 38, R <= 38, true}
           : G == 4  ? IterationForm{false, false, R >= 56}
           : G == 8  ? IterationForm{false, false, true}
           : G == 16 ? IterationForm{R <= 48, false, false}
                     : IterationForm{R <= 48, false, true};
}

// Kernel flags: diagnostic outputs, MAD scale instead of Eq. 1, the min form of
// Eq. 2's sign select (uses_min_form).  Each form has kernels of its own: with
// both in one kernel the schedule of either loop moved by up to 4 % with the
// other's.
enum : int { kFlagDiag = 1, kFlagMad = 2, kFlagMin = 4 };

// Whether a select may pick a positive sample by its bit patterns
// (select_rank).  That pass is the shorter one, but the min form's loops of 8
// lanes up to 46 slots and of long 2-lane windows are scheduled better without
// it (alpha = 10, 300 curves at W = 361, (8,46,2): 2.781 -> 2.729 ms; 495 curves
// at W = 121, (2,62,2): 1.568 -> 1.533; 618 at W = 97, (2,52,2): 1.674 -> 1.638).
// The other variants measured lose up to 2 % without it; (2,44), (8,24) and (8,40),
// which were not, lie on their side by lanes and slots alone.
__host__ __device__ constexpr bool picks_by_bits(int G, int R, int flags)
{
    return (flags & kFlagMin) == 0 || !((G == 8 && R <= 46) || (G == 2 && R > 38));
}

// Load the window of tile position q into registers: slot s = glane + G*i
// holds tile[q + s] for s < W, kGap past W.  Slots are stored in pairs
// (i = 2k, 2k+1 in x[k].x, x[k].y) for the packed FP32x2 arithmetic.
// `tail_only` (uniform) says that G*(R-2) <= W, so only the last register pair
// can hold slots past W; the general path re-derives each row's limit from an
// opaque register so the compiler does not keep R loop-invariant predicates
// alive across the chain.
template <int G, int R>
__device__ __forceinline__ void load_window(float2 (&x)[R / 2], const TileRef tile, int q, int glane,
                                            int W, bool tail_only)
{
    const int base = q + glane;
    if (tail_only) {
#pragma unroll
        for (int k = 0; k < R / 2 - 1; ++k) {
            x[k].x = tile[base + G * (2 * k)];
            x[k].y = tile[base + G * (2 * k + 1)];
        }
        const float a = tile[base + G * (R - 2)];
        const float b = tile[base + G * (R - 1)];
        x[R / 2 - 1].x = (glane + G * (R - 2) < W) ? a : kGap;
        x[R / 2 - 1].y = (glane + G * (R - 1) < W) ? b : kGap;
    } else {
        int lim = W - glane;  // slot row i is valid for this lane iff G*i < lim
        asm volatile("" : "+r"(lim));
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            const float a = tile[base + G * (2 * k)];
            const float b = tile[base + G * (2 * k + 1)];
            x[k].x = (G * (2 * k) < lim) ? a : kGap;
            x[k].y = (G * (2 * k + 1) < lim) ? b : kGap;
        }
    }
}

// Per-group median state carried along a chain.
struct MedianState {
    float m;   // current median (valid when `have`)
    int L;     // valid samples < m
    int E;     // samples == m
    int Gp;    // samples > m
    int nv;    // valid samples in the window
    bool have;
};

// The |t| form of the sign select serves 1/4 <= alpha <= 4 (process_chain).
__host__ __device__ inline bool uses_min_form(float alpha) { return !(alpha >= 0.25f && alpha <= 4.f); }

// The kernel build a curve needs (without kFlagDiag).
__host__ __device__ inline int curve_flavour(const Curve &c)
{
    return (c.scale_mode != 0 ? kFlagMad : 0) | (uses_min_form(c.alpha) ? kFlagMin : 0);
}

// Narrow groups (G <= 4 lanes per window) stage their trend values in the
// warp's shared-memory slice and write trend and detrended flux at the end of
// the tile, coalesced: their 32/G groups walk chains a whole chain apart, so a
// direct store from every group would touch 32/G separate DRAM sectors with
// 4 bytes each.  The slice then holds T more floats after the staged samples.
__host__ __device__ constexpr bool stages_outputs(int G) { return G <= 4; }

// Two consecutive windows of a chain finish together in the 32-lane variants
// of few slots: a lone window leaves the warp waiting for its reductions (ten
// shuffles and a quotient per iteration against six slot pairs of work).
// Together the two give the scheduler independent work, and their four sums
// share one tree: each halving step keeps half of the sums per lane, so eight
// shuffles serve both windows.  One curve of 18,000 samples at W = 361: 21.2 us,
// 24.2 one window at a time.
__host__ __device__ constexpr bool pairs_windows(int G, int R, int flags)
{
    return G == 32 && R <= 12 && (flags & kFlagMad) == 0;
}

// A window past Phase 1: its median, above-median count and output position.
struct Pending {
    float m;
    float centre;
    int gp;
    int nv;
    int64_t p;
    bool produce;
};

// The 32-lane sum of a in lanes 0-15 and of b in lanes 16-31.
__device__ __forceinline__ float half_sums(float a, float b, bool upper)
{
    float v = (upper ? b : a) + __shfl_xor_sync(0xffffffffu, upper ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Phases 2 and 3 of two windows whose residuals y = x - m are in ya and yb.
// Lanes 0-15 own window a, lanes 16-31 window b.
template <int R, int FLAGS>
__device__ __forceinline__ void finish_pair(const Curve &cv, const Diag &dg, const float2 (&ya)[R / 2],
                                            const float2 (&yb)[R / 2], const Pending &a, const Pending &b,
                                            float rho, float k1, int lane)
{
    constexpr bool abs_form = (FLAGS & kFlagMin) == 0;
    const bool upper = (lane & 16) != 0;
    const Pending own = upper ? b : a;
    float mu = own.m, s = 0.f;
    if (__any_sync(0xffffffffu, own.produce)) {
        float2 sa = make_float2(0.f, 0.f), sb = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < R / 2; ++k) {
            const float2 pa = make_float2(fmaxf(ya[k].x, 0.f), fmaxf(ya[k].y, 0.f));
            const float2 pb = make_float2(fmaxf(yb[k].x, 0.f), fmaxf(yb[k].y, 0.f));
            sa = __ffma2_rn(pa, pa, sa);
            sb = __ffma2_rn(pb, pb, sb);
        }
        const float s2 = half_sums(sa.x + sa.y, sb.x + sb.y, upper);
        const float msq = own.gp > 0 ? __fdividef(s2, (float)own.gp) : 0.f;
        s = kScaleFactor * sqrtf(msq);  // for the diagnostic output
        const bool iterate = own.produce && msq > 0.f;
        if (__any_sync(0xffffffffu, iterate)) {
            const float r = (msq >= 0x1p-126f) ? rsqrtf(msq) : 1.f / sqrtf(msq);
            const float kp = r * k1, kp_o = __shfl_xor_sync(0xffffffffu, kp, 16);
            const float ka = upper ? kp_o : kp, kb = upper ? kp : kp_o;
            const float2 ka2 = make_float2(ka, ka), kb2 = make_float2(kb, kb);
            const float na = cv.alpha * ka, nb = cv.alpha * kb;
            const float2 na2 = make_float2(na, na), nb2 = make_float2(nb, nb);
            const float2 rho2 = make_float2(rho, rho);
            float delta = 0.f, da = 0.f, db = 0.f;
#pragma unroll 1
            for (int it = 0; it < cv.iters; ++it) {
                float2 wa = make_float2(0.f, 0.f), wya = wa, wb = wa, wyb = wa;
                // u_eff^2 as in the one-window form below.
                auto slot = [&](const float2 y, float2 &w, float2 &wy, const float2 v, const float2 u) {
                    const float2 z = make_float2(fma_sat(-u.x, v.x, 1.f), fma_sat(-u.y, v.y, 1.f));
                    const float2 zz = __fmul2_rn(z, z);
                    w = __fadd2_rn(w, zz);
                    wy = __ffma2_rn(zz, y, wy);
                };
                if constexpr (abs_form) {
                    const float2 ca = make_float2(-da * ka, -da * ka), cb = make_float2(-db * kb, -db * kb);
#pragma unroll
                    for (int k = 0; k < R / 2; ++k) {
                        const float2 ta = __ffma2_rn(ya[k], ka2, ca), tb = __ffma2_rn(yb[k], kb2, cb);
                        slot(ya[k], wa, wya, __ffma2_rn(rho2, make_float2(fabsf(ta.x), fabsf(ta.y)), ta), ta);
                        slot(yb[k], wb, wyb, __ffma2_rn(rho2, make_float2(fabsf(tb.x), fabsf(tb.y)), tb), tb);
                    }
                } else {
                    const float2 ca = make_float2(-da * ka, -da * ka), cb = make_float2(-db * kb, -db * kb);
                    const float2 ea = make_float2(-da * na, -da * na), eb = make_float2(-db * nb, -db * nb);
#pragma unroll
                    for (int k = 0; k < R / 2; ++k) {
                        const float2 pa = __ffma2_rn(ya[k], ka2, ca), qa = __ffma2_rn(ya[k], na2, ea);
                        const float2 pb = __ffma2_rn(yb[k], kb2, cb), qb = __ffma2_rn(yb[k], nb2, eb);
                        const float2 ua = make_float2(fminf(pa.x, qa.x), fminf(pa.y, qa.y));
                        const float2 ub = make_float2(fminf(pb.x, qb.x), fminf(pb.y, qb.y));
                        slot(ya[k], wa, wya, ua, ua);
                        slot(yb[k], wb, wyb, ub, ub);
                    }
                }
                // Lane bit 4 picks the window, bit 3 sum(w) or sum(w y).
                const float fa = wa.x + wa.y, ga = wya.x + wya.y, fb = wb.x + wb.y, gb = wyb.x + wyb.y;
                const float f = (upper ? fb : fa) + __shfl_xor_sync(0xffffffffu, upper ? fa : fb, 16);
                const float g = (upper ? gb : ga) + __shfl_xor_sync(0xffffffffu, upper ? ga : gb, 16);
                const bool second = (lane & 8) != 0;
                float v = (second ? g : f) + __shfl_xor_sync(0xffffffffu, second ? f : g, 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                const float v_o = __shfl_xor_sync(0xffffffffu, v, 8);
                const float sw = second ? v_o : v, swy = second ? v : v_o;
                if (sw > 0.f) delta = __fdividef(swy, sw);
                const float d_o = __shfl_xor_sync(0xffffffffu, delta, 16);
                da = upper ? d_o : delta;
                db = upper ? delta : d_o;
            }
            if (iterate) mu = own.m + delta;
        }
    }
    if ((lane & 15) == 0 && own.p < cv.n) {
        const float nanv = __int_as_float(0x7fc00000);
        cv.trend[own.p] = own.produce ? mu : nanv;
        cv.detr[own.p] = own.produce ? __fdiv_rn(own.centre, mu) : nanv;
        if constexpr ((FLAGS & kFlagDiag) != 0) {
            if (dg.median) dg.median[own.p] = (own.nv >= 1) ? own.m : nanv;
            if (dg.nvalid) dg.nvalid[own.p] = own.nv;
            if (dg.nplus) dg.nplus[own.p] = (own.nv >= 1) ? own.gp : 0;
            if (dg.scale) dg.scale[own.p] = own.produce ? s : nanv;
        }
    }
}

template <int G, int R, int FLAGS>
__device__ __forceinline__ void process_chain(const Curve &cv, const Diag &dg, const TileRef tile,
                                              float *out, int64_t t0, int q0, int P, int glane)
{
    constexpr int S = G * R;
    const int W = cv.W;
    const int h = (W - 1) >> 1;
    const float alpha = cv.alpha;
    const float cst = cv.c;
    // Sign select of Eq. 2 through |t| (Phase 3): rho = (1 - alpha^2)/(1 +
    // alpha^2) and sigma = sqrt((1 + alpha^2)/2)/(c s).  The branch on the
    // small side is t (1 - |rho|), a difference, so rho's rounding (at most 3
    // units of roundoff) grows by (a^2 - 1)/2 there, a = max(alpha, 1/alpha).
    // This form serves 1/4 <= alpha <= 4, where u_eff^2 stays within
    // 4 + 1.5 (a^2 - 1) units of its value for the window's sigma (1.6e-6
    // relative at a = 4); every other alpha takes the min of two scaled
    // residuals.  With r = 1/sqrt(msq) (Phase 2), sigma = r k1 in that form,
    // and in the other kp = r k1, kn = alpha kp (k1 negated when alpha < 1).
    constexpr bool abs_form = (FLAGS & kFlagMin) == 0;
    const float rho = fmaf(-alpha, alpha, 1.f) / fmaf(alpha, alpha, 1.f);
    const float k1 = (abs_form ? sqrtf(0.5f * fmaf(alpha, alpha, 1.f)) : (alpha >= 1.f ? 1.f : -1.f)) /
                     (kScaleFactor * cst);
    const int iters = cv.iters;
    const bool tail_only = G * (R - 2) <= W;  // rows 0..R-3 hold only slots < W
    static_assert(R % 2 == 0, "slots are processed in pairs");
    float2 x[R / 2];
    MedianState st;
    st.m = 0.f;
    st.L = st.E = st.Gp = 0;
    st.nv = 0;
    st.have = false;
    float mad = 0.f;  // the last window's MAD (kFlagMad)
    float2 xh[pairs_windows(G, R, FLAGS) ? R / 2 : 1];  // the pair's first window
    Pending held{};

    int q = q0 - 1, left = P;
    bool begin = true;
#pragma unroll 1
    for (; left > 0; --left) {
        ++q;
        const int64_t p = t0 + q;

        // ---- slide: one sample leaves, one enters --------------------------
        if (!begin) {
            const float out = tile[q - 1];
            const float in = tile[q + W - 1];
            const bool ov = out > kGapLimit;
            const bool iv = in > kGapLimit;
            st.nv += (int)iv - (int)ov;
            if (st.have) {
                if (ov) {
                    if (out < st.m) --st.L;
                    else if (out == st.m) --st.E;
                    else --st.Gp;
                }
                if (iv) {
                    if (in < st.m) ++st.L;
                    else if (in == st.m) ++st.E;
                    else ++st.Gp;
                }
            }
        }

        load_window<G, R>(x, tile, q, glane, W, tail_only);

        if (begin) {
            begin = false;
            int c = 0;
#pragma unroll
            for (int k = 0; k < R / 2; ++k)
                c += ((x[k].x > kGapLimit) ? 1 : 0) + ((x[k].y > kGapLimit) ? 1 : 0);
            st.nv = group_sum_int<G>(c);
        }
        if (st.nv == 0) st.have = false;
        const int k = (st.nv - 1) >> 1;  // rank of the lower median among valid samples
        const bool need_full = (st.nv >= 1) && !st.have;
        // 0 = median unchanged, +1 = moves to the largest sample below m,
        // -1 = moves to the smallest sample above m.
        int move = 0;
        if (st.have) {
            if (k < st.L) move = 1;
            else if (k >= st.L + st.E) move = -1;
        }

        // ---- exact selection (chain start / restart) -----------------------
        if (__any_sync(0xffffffffu, need_full)) {
            // Rank k of the valid samples is rank (S - nv) + k of all S
            // slots: missing samples and the slots past W hold kGap, below
            // every sample.
            float mn = INFINITY, mx = -INFINITY;
#pragma unroll
            for (int k2 = 0; k2 < R / 2; ++k2) {
                const float a = x[k2].x, b = x[k2].y;
                mn = fminf(mn, fminf(a > kGapLimit ? a : INFINITY, b > kGapLimit ? b : INFINITY));
                mx = fmaxf(mx, fmaxf(a, b));
            }
            mn = -group_max<G>(-mn);
            mx = group_max<G>(mx);
            int le;
            bool below;
            const float mf = select_rank<G, R, false, picks_by_bits(G, R, FLAGS)>(
                x, need_full, mn == 0.f ? 0x7fffffffu : float_key(mn), mx == 0.f ? 0x80000000u : float_key(mx),
                S - st.nv, S, (S - st.nv) + k, 0.f, 0.f, &le, &below);
            float2 ef = make_float2(0.f, 0.f);  // 0/1 flags, exact below 2^24
#pragma unroll
            for (int k2 = 0; k2 < R / 2; ++k2)
                ef = __fadd2_rn(ef, make_float2(eq_flag(x[k2].x, mf), eq_flag(x[k2].y, mf)));
            const int ce = group_sum_int<G>((int)(ef.x + ef.y));
            if (need_full) {
                st.m = mf;
                st.L = below ? k : le - ce - (S - st.nv);
                st.E = ce;
                st.Gp = st.nv - st.L - st.E;
                st.have = true;
            }
        }

        // ---- one-rank move of the median -----------------------------------
        if (__any_sync(0xffffffffu, move != 0)) {
            // The two passes are built so that half their work runs on the
            // FMA pipe, which is otherwise idle here: a 0/1 float flag marks
            // slots at or above sm, one FFMA2 pushes them 2^127 down (slots
            // below keep their exact value), and ties are counted as float
            // sums of 0/1 flags (exact: at most S < 2^24).
            const float sg = (move < 0) ? -1.f : 1.f;
            const float2 sg2 = make_float2(sg, sg);
            const float sm = sg * st.m;
            const float2 push = make_float2(-0x1p127f, -0x1p127f);
            // Even and odd pairs keep separate maxima and tie counts (exact in
            // any order), which halves the dependent chains of both scans.
            float best0 = -INFINITY, best1 = -INFINITY;
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                const float2 y = __fmul2_rn(x[k], sg2);
                const float2 f = make_float2(ge_flag(y.x, sm), ge_flag(y.y, sm));
                const float2 yb = __ffma2_rn(f, push, y);
                if (k & 1) best1 = fmaxf(best1, fmaxf(yb.x, yb.y));
                else best0 = fmaxf(best0, fmaxf(yb.x, yb.y));
            }
            float best = group_max<G>(fmaxf(best0, best1));
            const float cand = sg * best;
            float2 ef0 = make_float2(0.f, 0.f), ef1 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                const float2 fl = make_float2(eq_flag(x[k].x, cand), eq_flag(x[k].y, cand));
                if (k & 1) ef1 = __fadd2_rn(ef1, fl);
                else ef0 = __fadd2_rn(ef0, fl);
            }
            const int e = group_sum_int<G>((int)((ef0.x + ef0.y) + (ef1.x + ef1.y)));
            if (move > 0) {
                st.Gp += st.E;
                st.L -= e;
                st.E = e;
                st.m = cand;
            } else if (move < 0) {
                st.L += st.E;
                st.Gp -= e;
                st.E = e;
                st.m = cand;
            }
        }

        // ---- Phases 2 and 3 -------------------------------------------------
        const float centre = tile[q + h];
        const bool produce = (p < cv.n) && (st.nv >= 1) && (st.nv >= cv.min_valid) &&
                             (centre > kGapLimit);
        if constexpr (pairs_windows(G, R, FLAGS)) {
            const float2 neg = make_float2(-st.m, -st.m);
#pragma unroll
            for (int k = 0; k < R / 2; ++k) x[k] = __fadd2_rn(x[k], neg);
            const Pending now{st.m, centre, st.Gp, st.nv, p, produce};
            // An odd chain's last window has no partner.
            const bool first = ((P - left) & 1) == 0;
            if (first) {
                held = now;
#pragma unroll
                for (int k = 0; k < R / 2; ++k) xh[k] = x[k];
                if (left > 1) continue;
            }
            const Pending none{0.f, 0.f, 0, 0, INT64_MAX, false};
            finish_pair<R, FLAGS>(cv, dg, xh, x, held, first ? none : now, rho, k1, glane);
            continue;
        }
        float mu = st.m;
        float s = 0.f;
        if (__any_sync(0xffffffffu, produce)) {
            const float m = st.m;
            const float2 negm = make_float2(-m, -m);
            float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < R / 2; ++k) {
                x[k] = __fadd2_rn(x[k], negm);  // y = x - m, exact sign
                const float2 yp = make_float2(fmaxf(x[k].x, 0.f), fmaxf(x[k].y, 0.f));
                s2 = __ffma2_rn(yp, yp, s2);
            }
            const float s2sum = group_sum<G>(s2.x + s2.y);
            // msq = S2 / n+ and s = 0.6745 sqrt(msq) (Eq. 1).  The iterations
            // take 1/(c s) as rsqrt(msq) / (0.6745 c): a fast quotient and an
            // approximate reciprocal square root, 2 ulp each, far below what
            // the trend resolves, in place of an IEEE quotient, root and
            // reciprocal.  A subnormal mean square takes the IEEE root.
            const float msq = (st.Gp > 0) ? __fdividef(s2sum, (float)st.Gp) : 0.f;
            s = kScaleFactor * sqrtf(msq);  // for the diagnostic output
            if constexpr ((FLAGS & kFlagMad) != 0) {
                // MAD = the order statistic of rank floor((nv-1)/2) of |y| over
                // the valid slots; gap slots have |y| near 2^100 and sort above
                // every candidate.  The search starts from the chain's last
                // MAD (at a chain start, from the scale of Eq. 1), where
                // ranks of |y| lie about s / (0.43 n) apart for normal
                // samples, and usually ends after two or three passes; a bit
                // by bit bisection took 30 per window (200 curves of 18,000
                // samples at W = 361: 6.87 ms, now 2.79).
                const float q0 = mad > 0.f ? mad : kScaleFactor * sqrtf(msq);
                int le;
                bool below;
                s = select_rank<G, R, true>(x, produce, 0u, __float_as_uint(0x1p98f), 0, st.nv,
                                            (st.nv - 1) >> 1, q0, __fdividef(q0, 0.43f * (float)st.nv), &le,
                                            &below);
                mad = produce ? s : 0.f;
            }
            const bool iterate = produce && ((FLAGS & kFlagMad) != 0 ? (s > 0.f) : (msq > 0.f));
            if (__any_sync(0xffffffffu, iterate)) {
                // Eq. 2 needs only u_eff^2 = k^2 (y - delta)^2 with k = kp =
                // 1/(c s) above the trend and k = kn = alpha/(c s) below it.
                // Eq. 4 in centred form: delta_new = sum(w y)/sum(w), since
                // mu = m + delta.
                float r;  // 0.6745 / s
                if constexpr ((FLAGS & kFlagMad) != 0) r = kScaleFactor / s;
                else r = (msq >= 0x1p-126f) ? rsqrtf(msq) : 1.f / sqrtf(msq);
                float delta = 0.f;
                if constexpr (abs_form) {
                    // t = sigma (y - delta), sigma^2 = (kp^2 + kn^2)/2:
                    // t (t + rho |t|) = kp^2 u^2 for u >= 0, kn^2 u^2 for u < 0,
                    // so one FMA with |t| as an operand does the sign select.
                    const float sg = r * k1;
                    const float2 sg2 = make_float2(sg, sg);
                    const float2 rho2 = make_float2(rho, rho);
#pragma unroll 1
                    for (int it = 0; it < iters; ++it) {
                        const float2 c0 = make_float2(-delta * sg, -delta * sg);
                        float2 swt = make_float2(0.f, 0.f), swyt = make_float2(0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < R / 2; ++k) {
                            constexpr IterationForm form = iteration_form(G, R);
                            const float2 ts = fma2<form.t>(x[k], sg2, c0);
                            const float2 v = fma2<form.v>(rho2, make_float2(fabsf(ts.x), fabsf(ts.y)), ts);
                            const float2 z = make_float2(fma_sat(-ts.x, v.x, 1.f), fma_sat(-ts.y, v.y, 1.f));
                            const float2 w = __fmul2_rn(z, z);
                            swt = __fadd2_rn(swt, w);
                            swyt = fma2<form.swy>(w, x[k], swyt);
                        }
                        const float sws = group_sum<G>(swt.x + swt.y);
                        const float swys = group_sum<G>(swyt.x + swyt.y);
                        // sws <= S, so the fast quotient (2 ulp) is safe here;
                        // its error is far below the FP32 rounding of the sums.
                        if (sws > 0.f) delta = __fdividef(swys, sws);
                    }
                } else {
                    // u_eff = min(y kp - delta kp, y kn - delta kn) when
                    // alpha >= 1 (max when alpha < 1; negating both keeps one
                    // code path).
                    const float kp = r * k1;
                    const float kn = alpha * kp;
                    const float2 kp2 = make_float2(kp, kp);
                    const float2 kn2 = make_float2(kn, kn);
#pragma unroll 1
                    for (int it = 0; it < iters; ++it) {
                        const float2 c1 = make_float2(-delta * kp, -delta * kp);
                        const float2 c2 = make_float2(-delta * kn, -delta * kn);
                        float2 swt = make_float2(0.f, 0.f), swyt = make_float2(0.f, 0.f);
#pragma unroll
                        for (int k = 0; k < R / 2; ++k) {
                            const float2 p1 = __ffma2_rn(x[k], kp2, c1);
                            const float2 p2 = fma2<true>(x[k], kn2, c2);
                            const float qa = fminf(p1.x, p2.x);
                            const float qb = fminf(p1.y, p2.y);
                            const float2 z = make_float2(fma_sat(-qa, qa, 1.f), fma_sat(-qb, qb, 1.f));
                            const float2 w = __fmul2_rn(z, z);
                            swt = __fadd2_rn(swt, w);
                            swyt = __ffma2_rn(w, x[k], swyt);
                        }
                        const float sws = group_sum<G>(swt.x + swt.y);
                        const float swys = group_sum<G>(swyt.x + swyt.y);
                        if (sws > 0.f) delta = __fdividef(swys, sws);
                    }
                }
                if (iterate) mu = m + delta;
            }
        }

        if (glane == 0 && p < cv.n) {
            const float nanv = __int_as_float(0x7fc00000);
            if constexpr (stages_outputs(G)) {
                out[q] = produce ? mu : nanv;  // written out by the tile's flush
            } else {
                cv.trend[p] = produce ? mu : nanv;
                cv.detr[p] = produce ? __fdiv_rn(centre, mu) : nanv;
            }
            if constexpr ((FLAGS & kFlagDiag) != 0) {
                if (dg.median) dg.median[p] = (st.nv >= 1) ? st.m : nanv;
                if (dg.nvalid) dg.nvalid[p] = st.nv;
                if (dg.nplus) dg.nplus[p] = (st.nv >= 1) ? st.Gp : 0;
                if (dg.scale) dg.scale[p] = produce ? s : nanv;
            }
        }
    }
}

// The curve that owns work item `item`: the last c with first_tile[c] <= item,
// by a warp-wide search that divides the range by 32 per round (two dependent
// loads for 1000 curves).  A table of items instead, 8 bytes per tile written
// by the host and copied before the launch, was 0.5 MB for 1000 curves of
// 18,000 samples, and grew with every shorter chain.
__device__ __forceinline__ int find_curve(const int32_t *__restrict__ first_tile, int n, int item, int lane)
{
    int lo = 0, len = n;
    while (len > 1) {
        const int step = (len + 31) >> 5;
        const int at = lane * step;
        const bool below = at < len && first_tile[lo + at] <= item;
        const int k = max(__popc(__ballot_sync(0xffffffffu, below)) - 1, 0);
        lo += k * step;
        len = min(step, len - k * step);
    }
    return lo;
}

// Work items belong to warps: each warp stages its own tile of T = (32/G)*P
// positions (plus the S-1 halo samples) in its slice of shared memory, so no
// CTA-wide barrier is ever needed.  Without a queue, warp w of CTA b takes
// item b*warps + w; with a queue, each warp pulls items until none is left.
// Every warp makes exactly one pull past the end, so the counter's wrap value
// brings it back to 0 with the launch's last pull and the next launch needs
// no memset before it.
// Dynamic shared memory: warps * (T + S - 1) floats, plus warps * T for the
// staged trend when stages_outputs(G).  MINB (CTAs of 256
// threads per SM) sets the register budget the compiler aims for.  FLAGS
// selects the diagnostic outputs, the MAD scale and the sign select's form;
// every curve of one launch must have the scale mode and an alpha that the
// kernel was built for (curve_flavour).  Pairs of windows need 79
// registers (at 64 they spill): 24 warps per SM.
template <int G, int R, int MINB, int FLAGS>
__global__ void __launch_bounds__(256, pairs_windows(G, R, FLAGS) ? 3 : MINB) umi_tile_kernel(LaunchArgs a)
{
    extern __shared__ float smem[];
    constexpr int S = G * R;
    // Launched as a programmatic dependent (see the launcher): nothing of
    // global memory is touched before the work ahead in the stream is done.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int n_warps = blockDim.x >> 5;
    const int glane = lane & (G - 1);
    const int group = lane / G;
    const int P = a.chain;
    const int T = (32 / G) * P;
    const int tile_len = T + S - 1;
    const int slice_len = tile_len + (stages_outputs(G) ? T : 0);
    float *tile = smem + (size_t)warp * slice_len;
    float *out = tile + tile_len;  // staged trend of the tile's positions (narrow groups)
#ifdef UMI_CHECKED
    {
        unsigned dsm;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dsm));
        if ((uint64_t)n_warps * (uint64_t)slice_len * sizeof(float) > dsm) {
            if (threadIdx.x == 0 && a.check) atomicOr(a.check, kCheckSmemSize);
            return;
        }
    }
    const TileRef tref{tile, tile_len, a.check};
#else
    const TileRef tref{tile};
#endif

    int item = blockIdx.x * n_warps + warp;
    for (;;) {
        if (a.queue) {
            int v = 0;
            if (lane == 0) v = (int)atomicInc(a.queue, (unsigned)a.n_items + gridDim.x * n_warps - 1u);
            item = __shfl_sync(0xffffffffu, v, 0);
        }
        if (item >= a.n_items) break;
        int curve = 0, tile_idx = item;
        if (a.curves) {
            curve = find_curve(a.first_tile, a.n_curves, item, lane);
#ifdef UMI_CHECKED
            if (curve < 0 || curve >= a.n_curves) {
                if (lane == 0 && a.check) atomicOr(a.check, kCheckCurveIndex);
                if (!a.queue) break;
                continue;
            }
#endif
            tile_idx -= a.first_tile[curve];
        }
        const Curve cv = a.curves ? a.curves[curve] : a.single;
        const int64_t t0 = (int64_t)tile_idx * T;
        const int h = (cv.W - 1) >> 1;
#ifdef UMI_CHECKED
        if (tile_idx < 0 || t0 >= (cv.n > 0 ? cv.n : 1)) {
            if (lane == 0 && a.check) atomicOr(a.check, kCheckItemTile);
            if (!a.queue) break;
            continue;
        }
#endif

        // Stage with asynchronous 4-byte copies (no alignment beyond the
        // float's), then turn the non-finite samples each lane copied into
        // the gap marker; slots outside the curve get it directly.
        for (int k = lane; k < tile_len; k += 32) {
            const int64_t idx = t0 - h + k;
            if (idx >= 0 && idx < cv.n) cp_async4(tile + k, cv.flux + idx);
            else tile[k] = kGap;
        }
        cp_async_wait_all();
        for (int k = lane; k < tile_len; k += 32)
            if (!isfinite(tile[k])) tile[k] = kGap;
        __syncwarp();
        process_chain<G, R, FLAGS>(cv, a.diag, tref, out, t0, group * P, P, glane);
        __syncwarp();  // every lane is done with the tile before it is restaged
        if constexpr (stages_outputs(G)) {
            // Flush: position k of the tile has its sample at tile[k + h];
            // a NaN trend (no estimate) gives a NaN quotient too.
            const float nanv = __int_as_float(0x7fc00000);
            const int kend = (int)min((int64_t)T, cv.n - t0);
            for (int k = lane; k < kend; k += 32) {
                const float mu = out[k];
                cv.trend[t0 + k] = mu;
                cv.detr[t0 + k] = (mu == mu) ? __fdiv_rn(tref[k + h], mu) : nanv;
            }
            __syncwarp();  // the flush reads the tile: done before it is restaged
        }
        if (!a.queue) break;
    }
}

}  // namespace umi
