// rs_segmented.cuh -- kernels of the segmented sort.
//
// A segmented sort sorts every segment [off[s], off[s+1]) of one array on its
// own (the paper has no segmented case; this is the plain definition applied
// per segment).  Segments are routed by size (rs_small.cuh has the first two):
//   tiny (2 <= size <= warp_max): k_bin_sort with a CTA of two warps per segment;
//   small (warp_max < size <= small_max): k_bin_sort (rs_bin_sort.cuh), one CTA
//       per segment, the whole segment on chip -- one read and one write of
//       every item either way;
//   large (size > small_max): scatter passes as of the unsegmented sort
//       (k_onesweep<..., SEG>) over tiles that never straddle a segment, after
//       k_seg_hist (per-segment digit histograms) and k_seg_scan (per-segment
//       bucket bases, and each segment's order: one pass by digit 3 and its
//       buckets sorted on chip, or all passes).
// k_seg_plan validates the table and lays the work out.
#pragma once

#include "rs_bin_sort.cuh"
#include "rs_device.cuh"

namespace rs {

// `count` threads write the tile geometries of one segment of `size` items from
// item `lo` on, tiles t0, t0 + 1, ...
__device__ __forceinline__ void write_tiles(uint4* tile_geo, uint32_t lo, uint32_t size,
                                            uint32_t t0, uint32_t ordinal, uint32_t tile,
                                            uint32_t thread, uint32_t count) {
    for (uint32_t k = thread; (unsigned long long)k * tile < size; k += count) {
        const uint32_t left = size - k * tile;
        tile_geo[t0 + k] = make_uint4(lo + k * tile, left < tile ? left : tile, t0, ordinal);
    }
}

// ---------------------------------------------------------------------------
// k_seg_plan: CTAs of 1024 threads, a segment per thread.
//  - Validates the table: nondecreasing, off[S] <= n, every segment < 2^30
//    items.  A bad table sets ERR_SEGMENTS; every later kernel then exits
//    without writing anything.
//  - Large segments get consecutive tile ids and a dense ordinal, in any order;
//    tile_geo[t] = (first item, item count, first tile of its segment, ordinal
//    of its segment).  Nothing is written past max_tiles or max_large, which a
//    bad table could ask for.
//  - Tiny and small segments are listed by size (list_small; order irrelevant).
//  - The pass plan runs all npass passes (four, or eight for 64-bit keys;
//    caller -> alternate -> ... -> caller), and the MSD-first pass of the segments
//    that take it.
// The order of segments does not matter to any later kernel, so CTAs take their
// places with one atomic each: 2^15 segments in 4 us, where one CTA that scanned
// over them in turn took 53.
// ---------------------------------------------------------------------------
static __global__ void __launch_bounds__(1024)
k_seg_plan(const uint32_t* __restrict__ off, uint32_t num_segments, uint32_t n, uint32_t tile,
           uint32_t warp_max, uint32_t small_max, Ctrl* __restrict__ ctrl,
           uint32_t* __restrict__ sticky, uint4* __restrict__ tile_geo, uint32_t max_tiles,
           uint32_t* __restrict__ tiny_list, uint32_t* __restrict__ small_list,
           uint32_t* __restrict__ large_first /* [S] first item of large ordinal */,
           uint32_t max_large, uint32_t npass = PASSES) {
    __shared__ unsigned long long s_w64[32];
    __shared__ uint32_t s_base[2];  // this CTA's first tile and first ordinal
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_launch_next();
    pdl_wait();

    const uint32_t s = blockIdx.x * 1024 + tid;
    uint32_t size = 0, lo = 0;
    bool bad = false;
    if (s < num_segments) {
        lo = off[s];
        const uint32_t hi = off[s + 1];
        bad = hi < lo || hi > n || hi - lo >= (1u << 30);
        size = bad ? 0u : hi - lo;
    }
    const bool large = size > small_max;
    const uint32_t ntiles = large ? (size + tile - 1) / tile : 0u;
    list_small(ctrl, s, large ? 0u : size, warp_max, num_segments - 1, tiny_list, small_list);
    // CTA-wide exclusive scan of (tiles, large flag), two 32-bit halves.
    const unsigned long long v = ((unsigned long long)ntiles << 32) | (large ? 1u : 0u);
    unsigned long long x = v;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w64[warp] = x;
    __syncthreads();
    unsigned long long before = 0, all = 0;
    for (uint32_t w = 0; w < 32; ++w) {
        if (w < warp) before += s_w64[w];
        all += s_w64[w];
    }
    if (tid == 0) {
        s_base[0] = atomicAdd(&ctrl->seg_tiles, (uint32_t)(all >> 32));
        s_base[1] = atomicAdd(&ctrl->large_count, (uint32_t)all);
        if (blockIdx.x == 0) {
            for (uint32_t p = 0; p < npass; ++p) ctrl->dir[p] = (p & 1) ? DIR_B_TO_A : DIR_A_TO_B;
            ctrl->dir[MSD_SLOT] = DIR_A_TO_B;
        }
    }
    __syncthreads();
    const unsigned long long excl = before + x - v;
    const uint32_t t0 = s_base[0] + (uint32_t)(excl >> 32);
    const uint32_t ordinal = s_base[1] + (uint32_t)excl;
    const bool fits = !large || (t0 + ntiles <= max_tiles && t0 + ntiles >= t0 &&
                                 ordinal < max_large);
    if (__any_sync(0xffffffffu, bad || !fits) && lane == 0)
        record_error(ctrl, sticky, ERR_SEGMENTS);
    if (large && fits) large_first[ordinal] = lo;
    // The warp writes the tiles of its large segments together.
    for (uint32_t todo = __ballot_sync(0xffffffffu, large && fits); todo != 0; todo &= todo - 1) {
        const uint32_t l = __ffs(todo) - 1;
        const uint32_t l_lo = __shfl_sync(0xffffffffu, lo, l);
        const uint32_t l_size = __shfl_sync(0xffffffffu, size, l);
        const uint32_t l_t0 = __shfl_sync(0xffffffffu, t0, l);
        const uint32_t l_ord = __shfl_sync(0xffffffffu, ordinal, l);
        write_tiles(tile_geo, l_lo, l_size, l_t0, l_ord, tile, lane, 32);
    }
}

// ---------------------------------------------------------------------------
// k_seg_hist: digit histograms of every large segment, added into
// hist[ordinal][4][256] (zeroed by the caller).  One CTA of 1024 threads per
// SM takes a contiguous run of tiles, so consecutive tiles mostly share a
// segment.  Counts accumulate in per-lane shared-memory columns (bin b of
// digit p as seen by lane l at word (p*256 + b)*32 + l: the 32 lanes of a warp
// always add into 32 different banks) and are summed into global memory only
// when the segment changes.  Also clears the first scatter pass's status
// array.  TYPED: keys are mapped onto their ordered words first.
// ---------------------------------------------------------------------------
constexpr uint32_t SEG_HIST_THREADS = 1024;
constexpr uint32_t SEG_HIST_COL_WORDS = PASSES * RADIX * 32;
constexpr uint32_t SEG_HIST_GEO_CHUNK = 1024;  // tile geometries staged at a time

template <bool TYPED>
__global__ void __launch_bounds__(SEG_HIST_THREADS, 1)
k_seg_hist(const uint32_t* __restrict__ keys, const Ctrl* __restrict__ ctrl,
           const uint4* __restrict__ tile_geo, uint32_t* __restrict__ hist,
           uint4* __restrict__ clear, uint32_t clear_vec4, uint32_t key_type) {
    extern __shared__ uint4 s_cols4[];
    uint32_t* const s_col = reinterpret_cast<uint32_t*>(s_cols4);
    constexpr uint32_t T = SEG_HIST_THREADS;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    pdl_launch_next();
    pdl_wait();  // the planner and the on-chip sorts are complete
    for (uint32_t i = blockIdx.x * T + tid; i < clear_vec4; i += gridDim.x * T)
        clear[i] = make_uint4(0, 0, 0, 0);
    if (ctrl->err != 0) return;
    const uint32_t tiles = ctrl->seg_tiles;
    const uint32_t per = (tiles + gridDim.x - 1) / gridDim.x;
    const uint32_t t_lo = blockIdx.x * per;
    const uint32_t t_hi = t_lo + per < tiles ? t_lo + per : tiles;
    if (t_lo >= t_hi) return;
    for (uint32_t i = tid; i < SEG_HIST_COL_WORDS / 4; i += T) s_cols4[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    uint32_t* const mycol = s_col + lane;
    auto count_key = [&](uint32_t k) {
        if (TYPED) k = key_to_ordered(k, key_type);
#pragma unroll
        for (uint32_t p = 0; p < PASSES; ++p)
            atomicAdd(mycol + ((p * RADIX + ((k >> (p * RADIX_BITS)) & (RADIX - 1))) << 5), 1u);
    };
    // Thread `bin` sums (and clears) the 32 columns of one bin, in rotated
    // order so that a warp's reads fall into 32 different banks.
    auto flush = [&](uint32_t seg) {
        __syncthreads();
        for (uint32_t bin = tid; bin < PASSES * RADIX; bin += T) {
            uint32_t c = 0;
#pragma unroll 8
            for (uint32_t j = 0; j < 32; ++j) {
                const uint32_t w = (bin << 5) + ((j + bin) & 31);
                c += s_col[w];
                s_col[w] = 0;
            }
            if (c) atomicAdd(hist + (size_t)seg * PASSES * RADIX + bin, c);
        }
        __syncthreads();
    };
    // Counts the keys [lo, hi): up to 3 before the first 16-byte boundary
    // and up to 3 after the last one one by one, the rest as 16-byte
    // vectors, four in flight per thread.
    auto count_range = [&](uint32_t lo, uint32_t hi) {
        const uint32_t* src = keys + lo;
        const uint32_t m = hi - lo;
        uint32_t head = (uint32_t)(((16u - ((uintptr_t)src & 15u)) & 15u) >> 2);
        if (head > m) head = m;
        const uint32_t nvec = (m - head) >> 2;
        const uint4* body = reinterpret_cast<const uint4*>(src + head);
        constexpr uint32_t LOADS = 4;
        for (uint32_t v = tid; v < nvec; v += LOADS * T) {
            uint4 x[LOADS];
#pragma unroll
            for (uint32_t u = 0; u < LOADS; ++u)
                if (v + u * T < nvec) x[u] = ld_stream(body + v + u * T);
#pragma unroll
            for (uint32_t u = 0; u < LOADS; ++u) {
                if (v + u * T < nvec) {
                    count_key(x[u].x), count_key(x[u].y);
                    count_key(x[u].z), count_key(x[u].w);
                }
            }
        }
        const uint32_t tail = head + nvec * 4;
        if (tid < head) count_key(ld_stream(src + tid));
        if (tid < 4 && tail + tid < m) count_key(ld_stream(src + tail + tid));
    };
    // The CTA's tiles, a chunk of geometries at a time in shared memory.
    // Consecutive tiles of one segment cover consecutive keys, so every run
    // of them is counted as one range (no per-tile wait on its geometry).
    __shared__ uint4 s_g[SEG_HIST_GEO_CHUNK];
    uint32_t cur = 0xffffffffu;
    for (uint32_t c0 = t_lo; c0 < t_hi; c0 += SEG_HIST_GEO_CHUNK) {
        const uint32_t cn = t_hi - c0 < SEG_HIST_GEO_CHUNK ? t_hi - c0 : SEG_HIST_GEO_CHUNK;
        __syncthreads();  // the previous chunk is no longer read
        for (uint32_t i = tid; i < cn; i += T) s_g[i] = tile_geo[c0 + i];
        __syncthreads();
        for (uint32_t ra = 0; ra < cn;) {
            const uint32_t seg = s_g[ra].w;
            uint32_t rb = ra;
            while (rb + 1 < cn && s_g[rb + 1].w == seg) ++rb;
            if (seg != cur) {
                if (cur != 0xffffffffu) flush(cur);
                cur = seg;
            }
            count_range(s_g[ra].x, s_g[rb].x + s_g[rb].y);
            ra = rb + 1;
        }
    }
    flush(cur);
}

// ---------------------------------------------------------------------------
// k_seg_scan: per large segment (one CTA of 1024 threads = 4 digits x 256
// buckets, twice for the eight digits of 64-bit keys), the exclusive prefix
// over buckets plus the segment's first item: the absolute first output slot
// of every bucket, written over the histogram hist[segment][NP][256].
//
// With route.geo set (32-bit keys), it also decides each segment's order: where
// digit 3 takes more than one value and no bucket of it holds more than
// MSD_SEG_BUCKET items, one pass by digit 3 into the alternate buffers, then runs
// of its buckets sorted on chip back into the caller's arrays; else the four
// passes.  Key-value segments whose digit 1 or 2 crowds (a bucket over four times its
// share) take the passes too: the on-chip sorts of their runs would take theirs (4096
// segments of 256 to 65536 pairs, ANDs of two words: 1670 us on chip, 1355 by the four
// passes; 256 distinct keys: 1480 and 1279; keys alone: 1204 and 1138, but 885 and 1136).
// Segments of the first kind get tiles 0 .. msd_tiles - 1 of route.geo, the others the
// lsd_tiles last ones; route.chunks lists (first item, items) of the runs: the buckets
// that start in the same stretch of CAPACITY - (largest bucket) items, CAPACITY in all
// at most.
// ---------------------------------------------------------------------------
constexpr uint32_t MSD_SEG_CAPACITY = SMALL_MID_MAX;  // of the on-chip sort
constexpr uint32_t MSD_SEG_BUCKET = MSD_SEG_CAPACITY - 512;  // so a stretch is 512 items or more

struct SegRoute {
    uint4* geo;
    uint2* chunks;
    uint32_t max_tiles, tile;
    bool pairs;
};

template <int NP = PASSES>
__global__ void __launch_bounds__(1024)
k_seg_scan(Ctrl* __restrict__ ctrl, uint32_t* __restrict__ hist,
           const uint32_t* __restrict__ large_first, const SegRoute route) {
    static_assert(NP == 4 || NP == 8, "32-bit or 64-bit keys");
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_max[PASSES * RADIX / 32], s_runs[RADIX / 32];  // by warps
    __shared__ uint32_t s_start[RADIX];      // first items of digit 3's buckets
    __shared__ uint32_t s_first[RADIX + 1];  // first items of the runs, and the segment's end
    __shared__ uint32_t s_base[2];           // first tile, first run
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t p = tid >> 8;
    pdl_launch_next();
    pdl_wait();  // the segment histograms are complete
    if (ctrl->err != 0) return;
    const uint32_t large = ctrl->large_count;
    for (uint32_t g = blockIdx.x; g < large; g += gridDim.x)
    for (uint32_t round = 0; round < NP / 4; ++round) {
        uint32_t* h = hist + ((size_t)g * NP + 4 * round) * RADIX;
        const uint32_t v = h[tid];
        uint32_t x = v;
#pragma unroll
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        const uint32_t most = __reduce_max_sync(0xffffffffu, v);
        if (lane == 0) s_max[warp] = most;
        __syncthreads();
        uint32_t offv = 0;
        for (uint32_t w = p * (RADIX / 32); w < warp; ++w) offv += s_warp[w];
        const uint32_t lo = large_first[g];
        const uint32_t start = offv + x - v;
        h[tid] = lo + start;
        if (NP == 4 && route.geo != nullptr) {
            constexpr uint32_t W = RADIX / 32;  // warps of a digit
            uint32_t size = 0, biggest = 0, big1 = 0, big2 = 0;
            for (uint32_t w = 0; w < W; ++w) {
                size += s_warp[w];  // digit 0 counts every item
                biggest = max(biggest, s_max[(PASSES - 1) * W + w]);
                big1 = max(big1, s_max[W + w]);
                big2 = max(big2, s_max[2 * W + w]);
            }
            // (A digit that is the same in all says nothing about the others.)
            const uint32_t crowd = size / RADIX * 4;
            const bool crowded = route.pairs && ((big1 > crowd && big1 < size) ||
                                                 (big2 > crowd && big2 < size));
            const bool msd = biggest <= MSD_SEG_BUCKET && biggest < size && !crowded;
            const uint32_t b = tid & (RADIX - 1);
            if (p == PASSES - 1) s_start[b] = start;
            __syncthreads();
            // Bucket b starts a run where its stretch is not that of the bucket
            // before (empty buckets start where the next one does).
            const uint32_t stretch = MSD_SEG_CAPACITY - (msd ? biggest : 0u);
            const bool starts = p == PASSES - 1 && msd &&
                                (b == 0 || start / stretch != s_start[b - 1] / stretch);
            const uint32_t vote = __ballot_sync(0xffffffffu, starts);
            if (p == PASSES - 1 && lane == 0) s_runs[warp & 7] = __popc(vote);
            __syncthreads();
            uint32_t at = __popc(vote & lanemask_lt()), runs = 0;
            for (uint32_t w = 0; w < RADIX / 32; ++w) {
                if (w < (warp & 7)) at += s_runs[w];
                runs += s_runs[w];
            }
            if (starts) s_first[at] = start;
            if (tid == 0) {
                s_first[runs] = size;
                const uint32_t tiles = (size + route.tile - 1) / route.tile;
                s_base[0] = msd ? atomicAdd(&ctrl->msd_tiles, tiles)
                                : route.max_tiles - tiles - atomicAdd(&ctrl->lsd_tiles, tiles);
                if (msd) s_base[1] = atomicAdd(&ctrl->chunk_count, runs);
            }
            __syncthreads();
            write_tiles(route.geo, lo, size, s_base[0], g, route.tile, tid, 1024);
            if (tid < runs)
                route.chunks[s_base[1] + tid] =
                    make_uint2(lo + s_first[tid], s_first[tid + 1] - s_first[tid]);
        }
        __syncthreads();
    }
}

}  // namespace rs
