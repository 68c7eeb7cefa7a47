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

// The open segment's first sample and the number of the curve's valid samples
// before it.
struct Open {
    int64_t start;  // -1: none
    int64_t rank;
};

__device__ __forceinline__ unsigned lanes_below(int lane) { return (1u << lane) - 1u; }

// Highest lane of `mask` (not 0).
__device__ __forceinline__ int top_lane(unsigned mask) { return 31 - __clz((int)mask); }

// Inclusive sum over the warp.
__device__ __forceinline__ int warp_scan(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

__device__ __forceinline__ int64_t tiles_of(int64_t len, int tile)
{
    return len < INT32_MAX / 2 ? (int64_t)(((uint32_t)len + (uint32_t)tile - 1u) / (uint32_t)tile)
                               : (len + tile - 1) / tile;
}

// One pass over a curve per CTA, 64 samples per thread at a time; each valid
// sample that follows a run of at least gap_min missing ones opens a segment and
// closes the one before it.  WRITE: put the kept segments into `table` and their
// first work items into `first_tile` (and clear the work counters); else count
// them.  Bound by latency, a chunk of samples waiting for the one before: so a
// thread's place among the others comes from ballots and one shuffle (positions
// ascend with the lane), every warp reads the other warps' totals itself instead
// of waiting for one that scans them, positions and counts inside a chunk are 32 bits, the
// next chunk's mask is loaded ahead, and words without a segment start skip the
// rest.  Two barriers per chunk to count, three to write.  A chunk of 65,536
// samples takes 1.9 us per pass (one curve of 1e8 samples; with four scans over
// the CTA's threads in shared memory 9.5): one curve of 1e7 samples at W = 25 3.38 -> 1.04 ms
// for the whole call (its mask scanned on the host 1.28), 256 Kepler curves of 4k
// to 70k 520 -> 490 us.
template <int WARPS, bool WRITE>
__global__ void __launch_bounds__(WARPS * 32)
    segment_scan_kernel(const unsigned *__restrict__ bits, const float *flux0,
                        const Curve *__restrict__ curves, const SegmentRule *__restrict__ rules,
                        SegmentCount *__restrict__ counts, Curve *__restrict__ table,
                        int32_t *__restrict__ first_tile, uint32_t *__restrict__ counters, int n_counters)
{
    constexpr int kChunk = 2048 * WARPS;
    __shared__ int2 sh_valid[WARPS];  // last valid sample (in the chunk, -1: none) and valid samples per warp
    __shared__ int2 sh_open[WARPS];   // last segment start (-1: none) and its rank in the chunk
    __shared__ int2 sh_kept[WARPS];   // kept segments and their tiles
    const Curve cv = curves[blockIdx.x];
    const SegmentRule r = rules[blockIdx.x];
    const int64_t first = cv.flux - flux0;  // the curve's first sample in the mask
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int at = threadIdx.x * 64;        // this thread's samples in the chunk
    int64_t last_valid = -1;                // carries, the same in every thread
    int64_t rank = 0;
    Open open{-1, 0};
    int64_t n_seg = 0, n_tiles = 0;         // WRITE: a carry too; else this thread's
    if constexpr (WRITE)
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_counters; k += gridDim.x * blockDim.x)
            counters[k] = 0u;

    // Takes the segment [start, end) holding `valid` samples if it is kept.
    auto close = [&](const Open &o, int64_t end, int64_t end_rank, auto &&kept) {
        if (o.start >= 0 && end_rank - o.rank >= r.min_seg) kept(o.start, end);
    };
    auto put = [&](int64_t start, int64_t end, int64_t seg, int64_t tiles) {
        Curve c = cv;
        c.flux += start;
        c.trend += start;
        c.detr += start;
        c.n = end - start;
        table[r.seg_base + seg] = c;
        first_tile[r.seg_base + seg] = (int32_t)(r.tile_base + tiles);
    };

    uint64_t word = validity_word(bits, first + at, first + cv.n);
    for (int64_t base = 0; base < cv.n; base += kChunk) {
        const uint64_t next = validity_word(bits, first + base + kChunk + at, first + cv.n);
        // The last valid sample and the valid samples before this word.
        const int own = word ? at + 63 - __clzll((long long)word) : -1;
        const unsigned some = __ballot_sync(0xffffffffu, word != 0);
        const unsigned some_below = some & lanes_below(lane);
        const int near = __shfl_sync(0xffffffffu, own, some_below ? top_lane(some_below) : 0);
        const int count = __popcll(word);
        const int upto = warp_scan(count, lane);
        int before_rel = some_below ? near : -1, rank_rel = upto - count;
        int chunk_last = some ? __shfl_sync(0xffffffffu, own, top_lane(some)) : -1;
        int chunk_rank = __shfl_sync(0xffffffffu, upto, 31);
        if constexpr (WARPS > 1) {
            if (lane == 0) sh_valid[warp] = make_int2(chunk_last, chunk_rank);
            __syncthreads();
            const int2 w = lane < WARPS ? sh_valid[lane] : make_int2(-1, 0);
            const unsigned full = __ballot_sync(0xffffffffu, w.x >= 0), full_below = full & lanes_below(warp);
            const int prev = __shfl_sync(0xffffffffu, w.x, full_below ? top_lane(full_below) : 0);
            if (!some_below && full_below) before_rel = prev;
            rank_rel += __reduce_add_sync(0xffffffffu, lane < warp ? w.y : 0);
            chunk_last = full ? __shfl_sync(0xffffffffu, w.x, top_lane(full)) : -1;
            chunk_rank = __reduce_add_sync(0xffffffffu, w.y);
        }
        const int64_t before = before_rel >= 0 ? base + before_rel : last_valid;

        // Visits this word's segment starts in order: sample, the end of the
        // segment before it, and its rank in the chunk.
        auto visit = [&](auto &&on_start) {
            int64_t lv = before;
            int seen = 0;
            uint64_t w = word;
            while (w) {
                const int bit = __ffsll((long long)w) - 1;
                const int64_t i = base + at + bit;
                if (lv < 0 || i - lv - 1 >= r.gap_min) on_start(at + bit, lv + 1, rank_rel + seen);
                // On to the end of this run of valid samples.
                const uint64_t inv = ~(w >> bit);
                const int run = min(inv ? __ffsll((long long)inv) - 1 : 64, 64 - bit);
                seen += run;
                lv = i + run - 1;
                w = bit + run < 64 ? (w >> (bit + run)) << (bit + run) : 0ull;
            }
        };
        // The open segment before this word: the last start before it.
        int2 mine = make_int2(-1, 0);
        visit([&](int start, int64_t, int rk) { mine = make_int2(start, rk); });
        const unsigned starts = __ballot_sync(0xffffffffu, mine.x >= 0);
        const unsigned starts_below = starts & lanes_below(lane);
        int2 pre = make_int2(-1, 0), all = make_int2(-1, 0);
        if (starts) {
            const int src = starts_below ? top_lane(starts_below) : 0, top = top_lane(starts);
            const int px = __shfl_sync(0xffffffffu, mine.x, src), py = __shfl_sync(0xffffffffu, mine.y, src);
            if (starts_below) pre = make_int2(px, py);
            all = make_int2(__shfl_sync(0xffffffffu, mine.x, top), __shfl_sync(0xffffffffu, mine.y, top));
        }
        if constexpr (WARPS > 1) {
            if (lane == 0) sh_open[warp] = all;
            __syncthreads();
            const int2 w = lane < WARPS ? sh_open[lane] : make_int2(-1, 0);
            const unsigned full = __ballot_sync(0xffffffffu, w.x >= 0), full_below = full & lanes_below(warp);
            if (full) {
                const int src = full_below ? top_lane(full_below) : 0, top = top_lane(full);
                const int px = __shfl_sync(0xffffffffu, w.x, src), py = __shfl_sync(0xffffffffu, w.y, src);
                if (!starts_below && full_below) pre = make_int2(px, py);
                all = make_int2(__shfl_sync(0xffffffffu, w.x, top), __shfl_sync(0xffffffffu, w.y, top));
            }
        }
        const Open before_word = pre.x >= 0 ? Open{base + pre.x, rank + pre.y} : open;
        // Closes the segments that end at this word's starts.
        auto closed = [&](auto &&kept) {
            if (mine.x < 0) return;
            Open o = before_word;
            visit([&](int start, int64_t end, int rk) {
                close(o, end, rank + rk, kept);
                o = Open{base + start, rank + rk};
            });
        };
        if constexpr (WRITE) {
            int seg = 0, tiles = 0;  // the host has checked that a band's tiles fit 32 bits
            closed([&](int64_t start, int64_t end) {
                ++seg;
                tiles += (int)tiles_of(end - start, r.tile);
            });
            const bool any = __any_sync(0xffffffffu, seg > 0);
            const int seg_upto = any ? warp_scan(seg, lane) : 0, tiles_upto = any ? warp_scan(tiles, lane) : 0;
            int64_t seg0 = n_seg + seg_upto - seg, tiles0 = n_tiles + tiles_upto - tiles;
            int seg_all = __shfl_sync(0xffffffffu, seg_upto, 31), tiles_all = __shfl_sync(0xffffffffu, tiles_upto, 31);
            if constexpr (WARPS > 1) {
                if (lane == 0) sh_kept[warp] = make_int2(seg_all, tiles_all);
                __syncthreads();
                const int2 w = lane < WARPS ? sh_kept[lane] : make_int2(0, 0);
                seg0 += __reduce_add_sync(0xffffffffu, lane < warp ? w.x : 0);
                tiles0 += __reduce_add_sync(0xffffffffu, lane < warp ? w.y : 0);
                seg_all = __reduce_add_sync(0xffffffffu, w.x);
                tiles_all = __reduce_add_sync(0xffffffffu, w.y);
            }
            if (seg > 0)
                closed([&](int64_t start, int64_t end) {
                    put(start, end, seg0, tiles0);
                    ++seg0;
                    tiles0 += tiles_of(end - start, r.tile);
                });
            n_seg += seg_all;
            n_tiles += tiles_all;
        } else {
            closed([&](int64_t start, int64_t end) {
                ++n_seg;
                n_tiles += tiles_of(end - start, r.tile);
            });
        }
        if (all.x >= 0) open = Open{base + all.x, rank + all.y};
        if (chunk_last >= 0) last_valid = base + chunk_last;
        rank += chunk_rank;
        word = next;
    }
    // The segment that the curve's end closes.
    if constexpr (WRITE) {
        if (threadIdx.x == 0)
            close(open, last_valid + 1, rank, [&](int64_t start, int64_t end) { put(start, end, n_seg, n_tiles); });
    } else {
        if (threadIdx.x == 0)
            close(open, last_valid + 1, rank, [&](int64_t start, int64_t end) {
                ++n_seg;
                n_tiles += tiles_of(end - start, r.tile);
            });
        __shared__ longlong2 sh_sum[WARPS];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            n_seg += __shfl_xor_sync(0xffffffffu, n_seg, o);
            n_tiles += __shfl_xor_sync(0xffffffffu, n_tiles, o);
        }
        if (lane == 0) sh_sum[warp] = make_longlong2(n_tiles, n_seg);
        __syncthreads();
        if (threadIdx.x == 0) {
            SegmentCount c{0, 0};
            for (int w = 0; w < WARPS; ++w) {
                c.tiles += sh_sum[w].x;
                c.segments += sh_sum[w].y;
            }
            counts[blockIdx.x] = c;
        }
    }
}

// Arguments of either pass.
struct ScanArgs {
    const unsigned *bits;
    const float *flux;
    const Curve *curves;
    const SegmentRule *rules;
    SegmentCount *counts;   // count pass
    Curve *table;           // write pass
    int32_t *first_tile;
    uint32_t *counters;
    int n_counters;
};

template <int WARPS, bool WRITE>
void launch_scan(int n_curves, cudaStream_t stream, const ScanArgs &a)
{
    segment_scan_kernel<WARPS, WRITE><<<n_curves, WARPS * 32, 0, stream>>>(
        a.bits, a.flux, a.curves, a.rules, a.counts, a.table, a.first_tile, a.counters, a.n_counters);
}

// One CTA per curve, whose chunk is 2,048 samples per warp: one warp up to two
// chunks, 8 up to two of theirs, else 32.  Short curves in small CTAs, because an
// SM holds more of them (200,000 curves of 60 samples: 13.4 ms by 1 warp, 14.4 by
// 8, 20.7 by 32), long ones in large ones (one of 70,000: 111, 82, 78 us; of 1e6: 677,
// 225, 167); 2,000 of 5,000 take 623, 625 and 688 us.
template <bool WRITE>
void scan_segments(int n_curves, int64_t longest, cudaStream_t stream, const ScanArgs &a)
{
    if (longest <= 4096) launch_scan<1, WRITE>(n_curves, stream, a);
    else if (longest <= 32768) launch_scan<8, WRITE>(n_curves, stream, a);
    else launch_scan<32, WRITE>(n_curves, stream, a);
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

    // The curves that can hold a kept segment, by band: segments are planned from
    // the whole curves' bands, as the plain batched call would plan them.
    BandSizes sizes;
    std::vector<Curve> curves;
    curves.reserve((size_t)B);
    int64_t longest = 0;
    for (int32_t b = 0; b < B; ++b) {
        const int64_t o = offsets[b], n = offsets[b + 1] - offsets[b];
        sizes[std::make_pair((int)W[b], p.scale_mode)] += n;
        if (n == 0 || n < (sp.min_seg >= 0 ? sp.min_seg : W[b] / 3)) continue;
        curves.push_back(make_curve(flux + o, trend + o, detr + o, n, W[b], p));
        longest = std::max(longest, n);
    }
    if (curves.empty()) {
        cudaError_t e = cudaMemsetAsync(trend, 0xff, sizeof(float) * (size_t)total, stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(detr, 0xff, sizeof(float) * (size_t)total, stream);
        return e == cudaSuccess ? UMI_OK : fail_cuda(e, "segment scan");
    }
    BatchLayout lay;
    st = build_layout(curves, &lay, &sizes, /*split=*/true);
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
        scan_segments<false>((int)C, longest, stream,
                             ScanArgs{d_bits, flux, d_curves, d_rules, d_counts, nullptr, nullptr, nullptr, 0});
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
        if (e == cudaSuccess) {
            scan_segments<true>((int)C, longest, stream,
                                ScanArgs{d_bits, flux, d_curves, d_rules, nullptr,
                                         reinterpret_cast<Curve *>(dev + sc.curve_off),
                                         reinterpret_cast<int32_t *>(dev + sc.tile_off),
                                         reinterpret_cast<uint32_t *>(dev + sc.counter_off),
                                         (int)out.bands.size()});
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
