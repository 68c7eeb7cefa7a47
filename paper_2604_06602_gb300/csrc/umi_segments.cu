// umi_segments.cu -- gap handling before the detrend.
//
// The paper lists gap handling as the pipeline step before detrending
// (Table 3's caption) and scales the minimum segment length to W/3
// (Section 4, Kepler Long-Cadence).  Reading used here: a curve splits at
// every run of at least `gap_min` consecutive missing samples (default W);
// leading and trailing missing runs belong to no segment; a segment with
// fewer than `min_seg` valid samples (default floor(W/3)) is dropped.  Each
// kept segment is detrended as a curve of its own, so no window reaches
// across a split, and positions outside kept segments get NaN.
//
// One ballot kernel packs the validity of every sample into a bitmask (1 bit
// per sample).  The scan of the mask runs on the device too, one CTA per
// curve, twice: it counts each curve's kept segments and their tiles, and,
// once the host has summed the counts (16 bytes per curve, one
// synchronisation, which also yields segments_out), it writes the segments
// straight into the curve table of the batched launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "umi_internal.h"

namespace umi {

struct SegmentRule {
    int64_t gap_min;  // missing-run length that splits
    int64_t min_seg;  // valid samples a kept segment holds at least
    int32_t tile;     // positions per work item of the curve's band
    int32_t seg_base;   // where the curve's segments go in the table (write pass)
    int32_t tile_base;  // and the first work item of the first of them
};

struct SegmentCount {
    int64_t tiles;
    int64_t segments;
};

namespace {

constexpr int kSegThreads = 1024;
constexpr int kSegWarps = kSegThreads / 32;
constexpr int kSegChunk = 64 * kSegThreads;  // one 64-sample word per thread

// bits[w] bit b = flux[32 w + b] is finite (bits past `total` are 0).
__global__ void validity_bits_kernel(const float *__restrict__ flux, int64_t total,
                                     unsigned *__restrict__ bits)
{
    const int64_t words = (total + 31) / 32;
    const int lane = threadIdx.x & 31;
    for (int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32; w < words;
         w += ((int64_t)gridDim.x * blockDim.x) / 32) {
        const int64_t i = w * 32 + lane;
        const bool ok = i < total && isfinite(flux[i]);
        const unsigned b = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) bits[w] = b;
    }
}

// Validity of samples [i, i + 64) of the whole buffer, 0 from `end` on.
// Words past the one that holds sample end - 1 are not read.
__device__ __forceinline__ uint64_t validity_word(const unsigned *__restrict__ bits, int64_t i, int64_t end)
{
    if (i >= end) return 0;
    const int64_t w = i >> 5, last = (end - 1) >> 5;
    const unsigned sh = (unsigned)(i & 31);
    const unsigned a = bits[w], b = w + 1 <= last ? bits[w + 1] : 0u, c = w + 2 <= last ? bits[w + 2] : 0u;
    uint64_t v = ((uint64_t)__funnelshift_r(b, c, sh) << 32) | __funnelshift_r(a, b, sh);
    if (end - i < 64) v &= (1ull << (end - i)) - 1;
    return v;
}

// Start of the open segment: its first sample and the number of valid samples
// of the curve before it.
struct Open {
    int64_t start;  // -1: none
    int64_t rank;
};

// Exclusive scans over the CTA's threads, seeded with `carry`; `carry` becomes
// the value past the last thread.  `sh` holds kSegWarps entries.
__device__ __forceinline__ int64_t scan_max(int64_t v, int64_t *sh, int64_t &carry)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = max(v, u);
    }
    if (lane == 31) sh[warp] = v;
    __syncthreads();
    int64_t before = carry, all = carry;
    for (int w = 0; w < kSegWarps; ++w) {
        if (w < warp) before = max(before, sh[w]);
        all = max(all, sh[w]);
    }
    __syncthreads();
    const int64_t u = __shfl_up_sync(0xffffffffu, v, 1);
    carry = all;
    return lane ? max(before, u) : before;
}

__device__ __forceinline__ int64_t scan_sum(int64_t v, int64_t *sh, int64_t &carry)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) sh[warp] = v;
    __syncthreads();
    int64_t before = carry, all = carry;
    for (int w = 0; w < kSegWarps; ++w) {
        if (w < warp) before += sh[w];
        all += sh[w];
    }
    __syncthreads();
    const int64_t u = __shfl_up_sync(0xffffffffu, v, 1);
    carry = all;
    return lane ? before + u : before;
}

// One pass over a curve per CTA, 65,536 samples at a time.  A thread holds the
// validity of 64 samples; each valid sample that follows a run of at least
// gap_min missing ones opens a segment and closes the one before it.  Bound
// by its four block scans per 65,536 samples (a few us), not by its bytes.
// WRITE: put the kept segments into `table` and their first work items into
// `first_tile`; else count them.  Copying the mask to the host and scanning it
// there took 1.2 ms of a 1.74 ms call on 256 Kepler curves of 4k to 70k
// samples; the whole call now takes 0.54 ms.
template <bool WRITE>
__global__ void __launch_bounds__(kSegThreads)
    segment_scan_kernel(const unsigned *__restrict__ bits, const float *flux0,
                        const Curve *__restrict__ curves, const SegmentRule *__restrict__ rules,
                        SegmentCount *__restrict__ counts, Curve *__restrict__ table,
                        int32_t *__restrict__ first_tile)
{
    __shared__ int64_t sh[kSegWarps];
    __shared__ Open sh_open[kSegWarps];
    const Curve cv = curves[blockIdx.x];
    const SegmentRule r = rules[blockIdx.x];
    const int64_t first = cv.flux - flux0;  // the curve's first sample in the mask
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t last_valid = -1;      // carries, the same in every thread
    int64_t rank = 0;
    Open open{-1, 0};
    int64_t n_seg = 0, n_tiles = 0;

    // Appends the segment [start, end) holding `valid` samples if it is kept.
    auto close = [&](int64_t start, int64_t end, int64_t valid, int64_t &seg, int64_t &tiles) {
        if (start < 0 || valid < r.min_seg) return;
        if constexpr (WRITE) {
            Curve c = cv;
            c.flux += start;
            c.trend += start;
            c.detr += start;
            c.n = end - start;
            table[r.seg_base + seg] = c;
            first_tile[r.seg_base + seg] = (int32_t)(r.tile_base + tiles);
        }
        ++seg;
        tiles += (end - start + r.tile - 1) / r.tile;
    };

    for (int64_t base = 0; base < cv.n; base += kSegChunk) {
        const int64_t b0 = base + (int64_t)threadIdx.x * 64;
        const uint64_t word = validity_word(bits, first + b0, first + cv.n);
        const int64_t before = scan_max(word ? b0 + 63 - __clzll((long long)word) : -1, sh, last_valid);
        const int64_t rank0 = scan_sum(__popcll(word), sh, rank);

        // Visits this word's segment starts in order, with the open segment
        // and the last valid sample before each.
        auto visit = [&](Open &o, auto &&on_start) {
            int64_t lv = before;
            int seen = 0;
            uint64_t w = word;
            while (w) {
                const int bit = __ffsll((long long)w) - 1;
                const int64_t i = b0 + bit;
                if (lv < 0 || i - lv - 1 >= r.gap_min) {
                    on_start(o, lv + 1, rank0 + seen);
                    o.start = i;
                    o.rank = rank0 + seen;
                }
                // On to the end of this run of valid samples.
                const uint64_t inv = ~(w >> bit);
                const int run = min(inv ? __ffsll((long long)inv) - 1 : 64, 64 - bit);
                seen += run;
                lv = i + run - 1;
                w = bit + run < 64 ? (w >> (bit + run)) << (bit + run) : 0ull;
            }
        };
        // The open segment before this thread's word: the last start of the
        // threads before it.
        Open mine{-1, 0};
        visit(mine, [](Open &, int64_t, int64_t) {});
        Open inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t us = __shfl_up_sync(0xffffffffu, inc.start, o);
            const int64_t ur = __shfl_up_sync(0xffffffffu, inc.rank, o);
            if (lane >= o && inc.start < 0) inc = Open{us, ur};
        }
        if (lane == 31) sh_open[warp] = inc;
        __syncthreads();
        Open pre = open, all = open;
        for (int w = 0; w < kSegWarps; ++w) {
            const Open o = sh_open[w];
            if (o.start < 0) continue;
            if (w < warp) pre = o;
            all = o;
        }
        __syncthreads();
        {
            const int64_t us = __shfl_up_sync(0xffffffffu, inc.start, 1);
            const int64_t ur = __shfl_up_sync(0xffffffffu, inc.rank, 1);
            if (lane && us >= 0) pre = Open{us, ur};
        }
        open = all;
        // Count this word's kept segments, then (write pass) place them.
        int64_t seg = 0, tiles = 0;
        auto count = [&](int64_t start, int64_t end, int64_t valid) {
            if (start < 0 || valid < r.min_seg) return;
            ++seg;
            tiles += (end - start + r.tile - 1) / r.tile;
        };
        Open o = pre;
        visit(o, [&](Open &p, int64_t end, int64_t rk) { count(p.start, end, rk - p.rank); });
        int64_t seg0 = scan_sum(seg, sh, n_seg);
        int64_t tiles0 = scan_sum(tiles, sh, n_tiles);
        if constexpr (WRITE) {
            o = pre;
            visit(o, [&](Open &p, int64_t end, int64_t rk) { close(p.start, end, rk - p.rank, seg0, tiles0); });
        }
    }
    if (threadIdx.x == 0) {
        close(open.start, last_valid + 1, rank - open.rank, n_seg, n_tiles);
        if constexpr (!WRITE) counts[blockIdx.x] = SegmentCount{n_tiles, n_seg};
    }
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

umi_status detrend_segmented(const float *flux, const int64_t *offsets, const int32_t *W, int32_t B,
                             const umi_params *params, const umi_segment_params *seg, float *trend,
                             float *detr, int64_t *segments_out, cudaStream_t stream)
{
    NvtxRange nvtx("umi detrend segmented");
    clear_error();
    if (segments_out) *segments_out = 0;
    umi_params p;
    umi_status st = check_params(params, &p);
    if (st != UMI_OK) return st;
    umi_segment_params sp;
    umi_default_segment_params(&sp);
    if (seg) sp = *seg;
    if (B < 0) return fail(UMI_ERR_INVALID_ARG, "B must be >= 0");
    if (B == 0) return UMI_OK;
    if (!offsets || !W) return fail(UMI_ERR_INVALID_ARG, "null offsets or W");
    if (offsets[0] != 0) return fail(UMI_ERR_INVALID_ARG, "offsets[0] must be 0");
    for (int32_t b = 0; b < B; ++b) {
        if (offsets[b + 1] < offsets[b]) return fail(UMI_ERR_INVALID_ARG, "offsets must be non-decreasing");
        if (W[b] < 1 || (W[b] % 2) == 0 || W[b] > umi_max_window())
            return fail(UMI_ERR_INVALID_ARG, "W[" + std::to_string(b) + "] must be odd and in range");
    }
    const int64_t total = offsets[B];
    if (total == 0) return UMI_OK;
    if (!flux || !trend || !detr) return fail(UMI_ERR_INVALID_ARG, "null buffer");

    // The whole curves, by band: segments are planned from the whole curves'
    // bands, as the plain batched call would plan them.
    std::vector<Curve> curves;
    curves.reserve((size_t)B);
    for (int32_t b = 0; b < B; ++b) {
        const int64_t o = offsets[b], n = offsets[b + 1] - offsets[b];
        if (n > 0) curves.push_back(make_curve(flux + o, trend + o, detr + o, n, W[b], p));
    }
    BatchLayout lay;
    st = build_layout(curves, &lay);
    if (st != UMI_OK) return st;
    for (const auto &band : lay.bands) {
        st = prepare_kernel(band.plan, band.flavour);
        if (st != UMI_OK) return st;
    }
    const size_t C = lay.curves.size();
    std::vector<SegmentRule> rules(C);
    for (const auto &band : lay.bands)
        for (int32_t k = band.first_curve; k < band.first_curve + band.n_curves; ++k) {
            const Curve &c = lay.curves[k];
            rules[k].gap_min = sp.gap_min > 0 ? sp.gap_min : c.W;
            // A kept segment holds at least its first sample.
            rules[k].min_seg = std::max<int64_t>(1, sp.min_seg >= 0 ? sp.min_seg : c.W / 3);
            rules[k].tile = band.plan.tile();
            rules[k].seg_base = rules[k].tile_base = 0;
        }

    // Count.  Staging and scratch: [curves][rules][counts], then the mask in
    // the scratch.
    keep_pool_memory();
    const size_t rule_off = up256(C * sizeof(Curve)), count_off = rule_off + up256(C * sizeof(SegmentRule));
    const size_t bits_off = count_off + up256(C * sizeof(SegmentCount));
    const int64_t words = (total + 31) / 32;
    const size_t scan_bytes = bits_off + sizeof(unsigned) * (size_t)words;
    PinnedStaging stage;
    st = stage.acquire(bits_off);
    if (st != UMI_OK) return st;
    memcpy(stage.p, lay.curves.data(), C * sizeof(Curve));
    memcpy(stage.p + rule_off, rules.data(), C * sizeof(SegmentRule));
    char *scan = nullptr;
    cudaError_t e = cudaMallocAsync((void **)&scan, scan_bytes, stream);
    if (e != cudaSuccess) return fail_cuda(e, "cudaMallocAsync (segment scan)");
    e = cudaMemcpyAsync(scan, stage.p, count_off, cudaMemcpyHostToDevice, stream);
    const Curve *d_curves = reinterpret_cast<const Curve *>(scan);
    SegmentRule *d_rules = reinterpret_cast<SegmentRule *>(scan + rule_off);
    SegmentCount *d_counts = reinterpret_cast<SegmentCount *>(scan + count_off);
    unsigned *d_bits = reinterpret_cast<unsigned *>(scan + bits_off);
    if (e == cudaSuccess) {
        const int64_t blocks = std::min<int64_t>((words * 32 + 255) / 256, 1 << 16);
        validity_bits_kernel<<<(int)blocks, 256, 0, stream>>>(flux, total, d_bits);
        segment_scan_kernel<false><<<(int)C, kSegThreads, 0, stream>>>(d_bits, flux, d_curves, d_rules, d_counts,
                                                                       nullptr, nullptr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(stage.p + count_off, d_counts, C * sizeof(SegmentCount), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = stage.mark(stream);
    // NaN everywhere while the host waits for the counts; kept segments are
    // overwritten by the batch below.
    if (e == cudaSuccess) e = cudaMemsetAsync(trend, 0xff, sizeof(float) * (size_t)total, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(detr, 0xff, sizeof(float) * (size_t)total, stream);
    if (e == cudaSuccess) e = stage.wait();
    if (e != cudaSuccess) {
        stage.release(stream);
        cudaFreeAsync(scan, stream);
        return fail_cuda(e, "segment scan");
    }

    // Sum the counts into each curve's place in the table.
    const SegmentCount *counts = reinterpret_cast<const SegmentCount *>(stage.p + count_off);
    BatchLayout out;
    int64_t kept = 0;
    for (const auto &src : lay.bands) {
        BatchLayout::Band band = src;
        band.first_curve = (int32_t)kept;
        int64_t segs = 0, tiles = 0;
        for (int32_t k = src.first_curve; k < src.first_curve + src.n_curves && st == UMI_OK; ++k) {
            rules[k].seg_base = (int32_t)(kept + segs);
            rules[k].tile_base = (int32_t)tiles;
            segs += counts[k].segments;
            tiles += counts[k].tiles;
            if (kept + segs > INT32_MAX || tiles > INT32_MAX) st = fail(UMI_ERR_INVALID_ARG, "too many work items");
        }
        if (st != UMI_OK) break;
        kept += segs;
        band.n_curves = (int32_t)segs;
        band.n_items = (int32_t)tiles;
        if (band.n_items > 0) out.bands.push_back(band);
    }
    if (segments_out && st == UMI_OK) *segments_out = kept;
    if (st != UMI_OK || kept == 0) {
        cudaFreeAsync(scan, stream);
        count_launches(2);
        return st;
    }

    // Write the table and launch its bands.
    const Scratch sc = scratch_layout((size_t)kept, out.bands.size());
    char *dev = nullptr;
    int launches = 0;
    e = cudaMallocAsync((void **)&dev, sc.bytes, stream);
    if (e == cudaSuccess) {
        memcpy(stage.p + rule_off, rules.data(), C * sizeof(SegmentRule));
        e = cudaMemcpyAsync(d_rules, stage.p + rule_off, C * sizeof(SegmentRule), cudaMemcpyHostToDevice, stream);
        stage.release(stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(dev + sc.counter_off, 0, sc.bytes - sc.counter_off, stream);
        if (e == cudaSuccess) {
            segment_scan_kernel<true><<<(int)C, kSegThreads, 0, stream>>>(
                d_bits, flux, d_curves, d_rules, nullptr, reinterpret_cast<Curve *>(dev + sc.curve_off),
                reinterpret_cast<int32_t *>(dev + sc.tile_off));
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) st = enqueue_bands(out, dev, sc, stream, &launches);
        cudaFreeAsync(dev, stream);
    }
    cudaFreeAsync(scan, stream);
    count_launches(launches + 3);
    if (e != cudaSuccess) return fail_cuda(e, "segment table");
    return st;
}

}  // namespace umi

extern "C" {

void umi_default_segment_params(umi_segment_params *sp)
{
    if (!sp) return;
    sp->gap_min = 0;
    sp->min_seg = -1;
}

umi_status umi_detrend_segmented(const float *flux_d, const int64_t *offsets_h, const int32_t *W_h,
                                 int32_t B, const umi_params *params, const umi_segment_params *seg,
                                 float *trend_d, float *detr_d, int64_t *segments_out, void *stream)
{
    return umi::detrend_segmented(flux_d, offsets_h, W_h, B, params, seg, trend_d, detr_d,
                                  segments_out, (cudaStream_t)stream);
}

}  // extern "C"
