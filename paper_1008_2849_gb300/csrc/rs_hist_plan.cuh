// rs_hist_plan.cuh -- the small kernels around the scatter passes:
//   k_hist4, k_hist4_cols, k_hist8  one read of the keys builds the histograms of
//            all four (eight) digits (the counting step of Sec. 3, for every
//            digit at once);
//   k_plan   exclusive prefix over the buckets of every digit (Sec. 3 "prefix
//            sum"; Alg. 2 PrefixSum), the order of the digits and the pass plan;
//   k_chunk_bounds  where the chunks of the top-digits order begin.
#pragma once

#include <type_traits>

#include "rs_device.cuh"

namespace rs {

// ---------------------------------------------------------------------------
// k_clear_ctrl: zeroes the control block, and `vecs` 16-byte words at `more` (the counts
// of segments).  The histogram kernel after it is its programmatic dependent, which reads
// the keys meanwhile and waits before it adds to the counts.  With a memset in its place,
// and the histogram after that, a call takes 2 to 3 us more: 2^20 keys 39.2 us instead of
// 37.0, 50021 pairs 30.5 instead of 28.2.
// ---------------------------------------------------------------------------
static __global__ void __launch_bounds__(1024)
k_clear_ctrl(uint4* __restrict__ ctrl, uint4* __restrict__ more, size_t vecs) {
    static_assert(sizeof(Ctrl) % sizeof(uint4) == 0, "whole vectors");
    pdl_launch_next();
    if (blockIdx.x == 0)
        for (uint32_t i = threadIdx.x; i < sizeof(Ctrl) / sizeof(uint4); i += 1024)
            ctrl[i] = make_uint4(0, 0, 0, 0);
    for (size_t i = (size_t)blockIdx.x * 1024 + threadIdx.x; i < vecs; i += gridDim.x * 1024u)
        more[i] = make_uint4(0, 0, 0, 0);
}

// ---------------------------------------------------------------------------
// k_hist4: H[p][b] for p = 0..3 in one pass over the keys, added into
// hist[p * 256 + b] (which the caller zeroes; k_clear_ctrl may still be at it when the
// other histogram kernels start).
//
// Keys are read as 16-byte vectors (a scalar head and tail handle a base that
// is only 4-byte aligned) into a CTA-private shared histogram, which is added
// to the global one at the end.  How a warp updates the shared histogram is
// a tuning choice (MODE):
//   HIST_ATOMIC   every lane adds 1 to its bin;
//   HIST_LEADER   lanes whose digit equals lane 0's are added as one group
//                 (cheap, and it removes the worst shared-memory serialisation
//                 when most keys share a digit), the others add 1 each;
//   HIST_MATCH    lanes are grouped by digit with one ballot per digit bit and
//                 the lowest lane of every group adds the group's size.
// The kernel also clears the look-back status array of the first scatter
// pass.
// ---------------------------------------------------------------------------
constexpr int HIST_ATOMIC = 0;
constexpr int HIST_LEADER = 1;
constexpr int HIST_MATCH = 2;
constexpr int HIST_COLUMNS = 3;  // k_hist4_cols

// TYPED: keys are mapped onto their ordered words (key_type) before counting;
// unsigned keys use the instances without the map.
template <int THREADS, int MODE, bool TYPED>
__global__ void __launch_bounds__(THREADS)
k_hist4(const uint32_t* __restrict__ keys, uint32_t n, uint32_t* __restrict__ hist,
        uint4* __restrict__ clear, uint32_t clear_vec4, uint32_t key_type) {
    __shared__ uint32_t s_h[PASSES * RADIX];
    const uint32_t tid = threadIdx.x;
    const uint32_t lane = tid & 31;
    for (uint32_t i = tid; i < PASSES * RADIX; i += THREADS) s_h[i] = 0;

    const uint32_t gtid = blockIdx.x * THREADS + tid;
    const uint32_t gsize = gridDim.x * THREADS;
    for (uint32_t i = gtid; i < clear_vec4; i += gsize) clear[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    uint32_t head = (uint32_t)(((16u - ((uintptr_t)keys & 15u)) & 15u) >> 2);
    if (head > n) head = n;
    const uint32_t body4 = (n - head) >> 2;
    const uint32_t tail = head + body4 * 4;
    const uint4* __restrict__ body = reinterpret_cast<const uint4*>(keys + head);

    auto count_key = [&](uint32_t key, bool ok) {
        if (TYPED) key = key_to_ordered(key, key_type);
#pragma unroll
        for (uint32_t p = 0; p < PASSES; ++p) {
            const uint32_t d = (key >> (p * RADIX_BITS)) & (RADIX - 1);
            uint32_t* bin = &s_h[p * RADIX + d];
            if (MODE == HIST_ATOMIC) {
                if (ok) atomicAdd(bin, 1u);
            } else if (MODE == HIST_LEADER) {
                const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
                const uint32_t same = __ballot_sync(0xffffffffu, ok && d == d0);
                if (ok) {
                    if (d != d0) atomicAdd(bin, 1u);
                    else if (lane == (uint32_t)(__ffs(same) - 1)) atomicAdd(bin, (uint32_t)__popc(same));
                }
            } else {
                const uint32_t peers = match_label<RADIX_BITS>(d) & __ballot_sync(0xffffffffu, ok);
                if (ok && lane == (uint32_t)(__ffs(peers) - 1)) atomicAdd(bin, (uint32_t)__popc(peers));
            }
        }
    };

    // Warp-uniform loop: every iteration a warp takes 2 x 32 consecutive
    // vectors, so all 32 lanes always take part in the warp votes.
    const uint32_t gwarp = gtid >> 5;
    const uint32_t nwarps = gsize >> 5;
    for (uint32_t c = gwarp * 64; c < body4; c += nwarps * 64) {
        const uint32_t i0 = c + lane, i1 = c + 32 + lane;
        const bool ok0 = i0 < body4, ok1 = i1 < body4;
        const uint4 v0 = ok0 ? ld_stream(body + i0) : make_uint4(0, 0, 0, 0);
        const uint4 v1 = ok1 ? ld_stream(body + i1) : make_uint4(0, 0, 0, 0);
        count_key(v0.x, ok0); count_key(v0.y, ok0); count_key(v0.z, ok0); count_key(v0.w, ok0);
        count_key(v1.x, ok1); count_key(v1.y, ok1); count_key(v1.z, ok1); count_key(v1.w, ok1);
    }
    // At most 3 keys before the first 16-byte boundary and 3 after the last.
    if (blockIdx.x == 0 && tid < 8) {
        const uint32_t i = tid < 4 ? tid : tail + (tid - 4);
        const bool ok = tid < 4 ? i < head : i < n;
        if (ok) {
            const uint32_t key = TYPED ? key_to_ordered(keys[i], key_type) : keys[i];
#pragma unroll
            for (uint32_t p = 0; p < PASSES; ++p)
                atomicAdd(&s_h[p * RADIX + ((key >> (p * RADIX_BITS)) & (RADIX - 1))], 1u);
        }
    }
    __syncthreads();
    for (uint32_t i = tid; i < PASSES * RADIX; i += THREADS) {
        const uint32_t c = s_h[i];
        if (c) atomicAdd(hist + i, c);
    }
}

// ---------------------------------------------------------------------------
// k_hist4_cols: the same histograms with private columns: bin b of digit p, as
// seen by lane l, lives at word (p*256 + b)*COLS + l % COLS.  With 32 columns
// (128 KiB, one CTA per SM) the 32 lanes of a warp always add into 32
// different banks (one shared-memory wavefront per warp-wide add, whatever
// the keys).  Eight columns (32 KiB) take up to four, but a quarter of the time
// to clear and to sum, which is what small arrays pay for.  Columns are
// summed (in rotated order, conflict-free) at the end.
// ---------------------------------------------------------------------------
template <int COLS>
constexpr uint32_t HIST_COL_WORDS = PASSES * RADIX * COLS;

template <int THREADS, int COLS, bool TYPED>
__global__ void __launch_bounds__(THREADS, 1)
k_hist4_cols(const uint32_t* __restrict__ keys, uint32_t n, uint32_t* __restrict__ hist,
             uint4* __restrict__ clear, uint32_t clear_vec4, uint32_t key_type) {
    extern __shared__ uint4 s_cols4[];
    uint32_t* const s_col = reinterpret_cast<uint32_t*>(s_cols4);
    const uint32_t tid = threadIdx.x;
    const uint32_t lane = tid & 31;
    pdl_launch_next();  // the plan kernel may launch; it waits for this one
    for (uint32_t i = tid; i < HIST_COL_WORDS<COLS> / 4; i += THREADS)
        s_cols4[i] = make_uint4(0, 0, 0, 0);
    const uint32_t gtid = blockIdx.x * THREADS + tid;
    const uint32_t gsize = gridDim.x * THREADS;
    for (uint32_t i = gtid; i < clear_vec4; i += gsize) clear[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    uint32_t head = (uint32_t)(((16u - ((uintptr_t)keys & 15u)) & 15u) >> 2);
    if (head > n) head = n;
    const uint32_t body4 = (n - head) >> 2;
    const uint32_t tail = head + body4 * 4;
    const uint4* __restrict__ body = reinterpret_cast<const uint4*>(keys + head);
    uint32_t* const mycol = s_col + lane % COLS;
    auto count_key = [&](uint32_t key) {
        if (TYPED) key = key_to_ordered(key, key_type);
#pragma unroll
        for (uint32_t p = 0; p < PASSES; ++p)
            atomicAdd(mycol + (p * RADIX + ((key >> (p * RADIX_BITS)) & (RADIX - 1))) * COLS, 1u);
    };
    // HIST_LOADS independent 16-byte loads in flight per thread and
    // iteration (64 KiB per SM): enough bytes in flight to cover the HBM
    // latency at full bandwidth.
    constexpr uint32_t HIST_LOADS = 4;
    for (uint32_t i = gtid; i < body4; i += HIST_LOADS * gsize) {
        uint4 v[HIST_LOADS];
#pragma unroll
        for (uint32_t u = 0; u < HIST_LOADS; ++u)
            v[u] = i + u * gsize < body4 ? ld_stream(body + i + u * gsize) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (uint32_t u = 0; u < HIST_LOADS; ++u) {
            if (i + u * gsize < body4) {
                count_key(v[u].x);
                count_key(v[u].y);
                count_key(v[u].z);
                count_key(v[u].w);
            }
        }
    }
    if (blockIdx.x == 0 && tid < 8) {
        const uint32_t i = tid < 4 ? tid : tail + (tid - 4);
        const bool ok = tid < 4 ? i < head : i < n;
        if (ok) count_key(keys[i]);
    }
    __syncthreads();
    pdl_wait();  // the counts are zero
    for (uint32_t bin = tid; bin < PASSES * RADIX; bin += THREADS) {
        uint32_t c = 0;
        const uint32_t turn = bin * COLS / 32 + bin;  // 32 lanes, 32 banks
#pragma unroll 8
        for (uint32_t j = 0; j < COLS; ++j) c += s_col[bin * COLS + (j + turn) % COLS];
        if (c) atomicAdd(hist + bin, c);
    }
}

// ---------------------------------------------------------------------------
// k_plan: G[p][b] = sum_{b' < b} H[p][b'] and the pass plan.  One CTA of
// 1024 threads, thread (p, b) = (tid / 256, tid % 256).  (Made by the histogram
// kernel's last CTA instead, it takes 4 us longer: as a kernel of its own it is
// resident when the counts are complete.)
//
// A pass whose digit takes one value for every key is the identity (a stable
// partition into one bucket).  Such passes are skipped, except that the
// number of executed passes is kept even (one trivial pass is run if needed)
// so that the ping-pong between the caller's arrays and the alternate
// buffers ends in the caller's arrays.
//
// MSD-first order (Alg. 2, "reverse sorting"), when msd_allowed: if digit 3
// is not trivial and no digit-3 bucket holds more than bucket_cap keys, the
// plan runs one pass by digit 3 (plan slot MSD_SLOT, caller's arrays ->
// alternate buffers) and skips passes 0..3; every bucket is then sorted on
// chip from the alternate buffers back into the caller's arrays (its digit 3
// is constant, so that pass is trivial there).  msd_off[b] is bucket b's
// first slot (msd_off[256] = n), and small_count becomes the number of buckets
// to sort (0 when the plan chooses the passes 0..3).
//
// Top-digits order, when top_bits > 0: if the keys spread evenly, only the
// passes by the two highest digits run.  The array is then stably sorted by
// its top 16 bits, and every chunk of keys with the same top_bits highest
// bits (about n >> top_bits of them) is sorted on chip by the rest.  "Evenly":
// no bucket of either digit holds over twice its share, at least three passes
// would run otherwise, and in a sample of the keys (the digits may be even one by one
// and not together)
//  - no chunk holds far more than its share: one hot key;
//  - the pairs of keys in one chunk are not far over those of even keys: few prefixes,
//    whose chunks are long (2^27 pairs with 10,000 prefixes 7.48 ms instead of 2.88);
//  - few keys are equal: chunks of repeated keys take the on-chip sorts longer (2^27 pairs
//    with 100,000 distinct keys 5.92 ms instead of 2.92, with 16 million 2.83 and 2.90).
// Chunks that are too long all the same are sorted in global memory by one CTA each, so a
// sample that misses them costs time, not correctness.
//
// 64-bit keys that are not even may still take the passes by their two to four highest
// digits that differ, if that saves two passes or more and the sample has no crowd of
// keys that these digits do not tell apart (normal doubles: three passes instead of
// eight).  Their chunks are chunk_step items long, up to the next change of prefix.
// ---------------------------------------------------------------------------
constexpr uint32_t TOP_MAX_SAMPLES = 8192;
constexpr uint32_t TOP_MAX_BITS = 16;

// Keys sampled: 8192 of 2^27 32-bit keys and more (repeated keys show by the sample's
// square over n; 3 us of 2.4 ms), else 4096.
__host__ __device__ constexpr uint32_t top_samples(uint32_t n, bool key64) {
    return !key64 && n >= (1u << 27) ? TOP_MAX_SAMPLES : 4096u;
}
// Times that every key may occur before the passes by all digits are the faster ones: 6 to
// 10 of 32-bit keys (2^25 to 2^27 of them, without or with values); of 64-bit keys 300 (2^22
// pairs), 50 (2^25).
__host__ __device__ constexpr uint32_t top_repeats(uint32_t n, bool key64) {
    return !key64 ? 8u : n >= (1u << 24) ? 48u : 192u;
}
// The least number of repeated keys in the sample that tells of so many times.  (64-bit
// arrays below 2^22 items are not looked at: it takes 5 us, and they gain 60.)
__host__ __device__ constexpr uint32_t top_equal_limit(uint32_t n, bool key64) {
    if (key64 && n < (1u << 22)) return ~0u;
    const unsigned long long s = top_samples(n, key64);
    const unsigned long long least = top_repeats(n, key64) * s * s / (2ull * n);
    return least < 2 ? 2u : least < s ? (uint32_t)least : (uint32_t)s;
}
// Samples of one key that tell of a chunk too long for one CTA to gain by: 0.1 % of 32-bit
// keys (2^25 pairs 879 us instead of 774 by all digits, with 0.05 % 773), 0.2 % of 64-bit.
__host__ __device__ constexpr uint32_t top_hot_limit(bool key64, uint32_t samples) {
    return samples / 4096 * (key64 ? 8 : 3);
}
// The most pairs of samples in one of 2^bits cells: four standard deviations over those of
// even keys, and those of cells whose sizes deviate by `spread` of their mean.
__device__ __forceinline__ uint32_t top_pair_limit(uint32_t samples, uint32_t bits,
                                                   float spread = 0.0f) {
    const uint32_t even = (uint32_t)((unsigned long long)samples * samples / 2 >> bits);
    return even + (uint32_t)(4.0f * sqrtf((float)even) + spread * spread * (float)even);
}

// What the plan works on; bucket_cap and msd_off for the MSD-first order
// (msd_off == nullptr: not allowed), top_bits for the top-digits order.
struct PlanArgs {
    Ctrl* ctrl;
    const void* keys;
    uint32_t n, key_type, bucket_cap;
    uint32_t* msd_off;
    uint32_t top_bits, chunk_step;
    uint32_t capacity;  // items of a chunk that a CTA takes
};

// Chunks are cut by prefix, so they grow longer where the keys are denser, and the top
// digit's histogram shows that better than a sample: this is how many items one of its
// values may have for its 2^(bits - 8) chunks to fit a CTA.  With over a sixteenth of the
// items in fuller ones an array takes the passes.  2^27 pairs whose density rises by 1.2, 1.5
// and 4 times from the least to the greatest key: 2497, 3843 and 5335 us by chunks, 2895 by
// the passes; 2^25 64-bit keys 1.2 and 2.1 times: 1184 and 2770 by prefix, 1128 by position.
__device__ __forceinline__ uint32_t top_digit_most(uint32_t bits, uint32_t capacity) {
    return (capacity - capacity / 64) << (bits - RADIX_BITS);
}

// Dynamic shared memory of k_plan when top_bits is set: two bytes for each cell of the
// 2^top_bits or 2^TOP_HASH_BITS, and where repeated keys are looked for at least a table of
// twice the samples with five bytes a slot.
constexpr uint32_t TOP_HASH_BITS = 13;
constexpr size_t top_plan_smem(uint32_t n, uint32_t top_bits, bool key64) {
    const size_t cells = sizeof(uint16_t) << (top_bits > TOP_HASH_BITS ? top_bits : TOP_HASH_BITS);
    const size_t samples = top_samples(n, key64);
    const size_t table = top_equal_limit(n, key64) < samples ? 5 * 2 * samples : 0;
    return cells > table ? cells : table;
}
constexpr size_t TOP_PLAN_SMEM = sizeof(uint16_t) << TOP_MAX_BITS;
static_assert(TOP_PLAN_SMEM >= 10 * TOP_MAX_SAMPLES, "the table too");
// TOP: the top-digits order may be chosen (without it the kernel is 4 KB of code, not 20).
template <int NPASS, bool TOP>
__global__ void __launch_bounds__(1024) k_plan(const PlanArgs plan) {
    extern __shared__ uint4 s_dyn[];
    static_assert(NPASS == 4 || NPASS == 8, "32-bit or 64-bit keys");
    using K = std::conditional_t<NPASS == 8, unsigned long long, uint32_t>;
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_trivial[NPASS];
    __shared__ uint32_t s_big, s_uneven, s_long;
    __shared__ uint32_t s_part[32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t b = tid & (RADIX - 1);
    Ctrl* const ctrl = plan.ctrl;
    const uint32_t n = plan.n, top_bits = TOP ? plan.top_bits : 0u;
    pdl_launch_next();
    pdl_wait();  // the histograms are complete
    if (tid < NPASS) s_trivial[tid] = 0;
    if (tid == 0) s_big = s_uneven = s_long = 0;
    // Thread (p, b): p = tid / 256 (+ 4 in the second round for 64-bit keys).
    uint32_t first3 = 0;  // digit 3, for the MSD-first order
    for (uint32_t round = 0; round < NPASS / 4; ++round) {
        const uint32_t p = (tid >> 8) + 4 * round;
        const uint32_t h = ctrl->hist[p][b];
        uint32_t x = h;
#pragma unroll
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        uint32_t off = 0;
        for (uint32_t w = (tid >> 8) * (RADIX / 32); w < warp; ++w) off += s_warp[w];
        const uint32_t first = off + x - h;
        ctrl->gofs[p][b] = first;
        if (h == n) s_trivial[p] = 1;
        if (p == PASSES - 1) {
            first3 = first;
            if (h > plan.bucket_cap) s_big = 1;
        }
        if (p >= NPASS - 2 && h > n / RADIX * 2) s_uneven = 1;
        if (TOP && p == NPASS - 1 && top_bits != 0 && h > top_digit_most(top_bits, plan.capacity))
            atomicAdd(&s_long, h);
        __syncthreads();  // s_warp is reused by the next round
    }
    const bool msd =
        NPASS == 4 && plan.msd_off != nullptr && !s_trivial[PASSES - 1] && !s_big;
    uint32_t executed = 0;
    for (uint32_t q = 0; q < NPASS; ++q) executed += s_trivial[q] ? 0 : 1;
    bool top = !msd && top_bits != 0 && !s_uneven && s_long <= n / 16 && executed >= 3;
    const bool deep = NPASS == 8 && top_bits != 0 && executed >= 4;
    uint32_t low = 0;  // the lowest digit with a pass
    if constexpr (TOP) if (top || deep) {  // the same for every thread
        uint32_t* const s_pair = reinterpret_cast<uint32_t*>(s_dyn);  // two 16-bit counts a word
        const K* const keys = static_cast<const K*>(plan.keys);
        constexpr uint32_t PER = NPASS == 4 ? TOP_MAX_SAMPLES / 1024 : 4;
        const uint32_t samples = top_samples(n, NPASS == 8);
        const uint32_t stride = n / samples;
        K k[PER];
#pragma unroll
        for (uint32_t q = 0; q < PER; ++q) {  // one key of each of `samples` parts
            const uint32_t i = q * 1024 + tid;
            uint32_t r = i * 0x9E3779B1u;
            r ^= r >> 15;
            r *= 0x85EBCA6Bu;
            const uint32_t at = (uint32_t)(((uint64_t)i * n) / samples) + __umulhi(r, stride);
            k[q] = i < samples ? key_to_ordered(keys[at], plan.key_type) : K(0);
        }
        // The sum of x over the threads (one barrier).
        auto sum_of = [&](uint32_t x) -> uint32_t {
            x = __reduce_add_sync(0xffffffffu, x);
            if (lane == 0) s_part[warp] = x;
            __syncthreads();
            return __reduce_add_sync(0xffffffffu, s_part[lane]);
        };
        // Keys that occur more than once in the sample, by a table of it (of 64-bit keys, of
        // 32 bits of their hashes), which holds all words but ~0.  One key that occurs
        // top_hot_limit times sets s_uneven.
        auto repeated_keys = [&]() -> uint32_t {
            constexpr uint32_t EMPTY = ~0u;
            const uint32_t slots = 2 * samples;  // a power of two
            uint32_t* const slot = s_pair;
            uint32_t* const again = s_pair + slots;  // a byte for each: its further samples
#pragma unroll 1
            for (uint32_t i = tid; i < slots * 5 / 16; i += 1024) {
                const uint32_t v = i < slots / 4 ? EMPTY : 0u;
                s_dyn[i] = make_uint4(v, v, v, v);
            }
            if (tid == 0) s_uneven = 0;
            __syncthreads();
            uint32_t found = 0;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                unsigned long long h = (unsigned long long)k[q] * 0x9E3779B97F4A7C15ull;
                h = (h ^ h >> 32) * 0xD6E8FEB86659FD93ull;
                const uint32_t word = NPASS == 4 ? (uint32_t)k[q] : (uint32_t)(h >> 32);
                if (q * 1024 + tid >= samples || word == EMPTY) continue;
                uint32_t at = (uint32_t)(h >> 16) & (slots - 1);
                uint32_t was = atomicCAS(&slot[at], EMPTY, word);
                // At most half of the slots are taken; a key that finds none is left out.
#pragma unroll 1
                for (uint32_t tries = 0; was != EMPTY && was != word && tries < 32; ++tries) {
                    at = (at + 1) & (slots - 1);
                    was = atomicCAS(&slot[at], EMPTY, word);
                }
                if (was != word) continue;
                // (A byte that overflows has passed the limit.)
                const uint32_t before =
                    atomicAdd(&again[at / 4], 1u << 8 * (at % 4)) >> 8 * (at % 4) & 0xffu;
                found += before == 0;
                if (before + 2 >= top_hot_limit(NPASS == 8, samples)) s_uneven = 1;
            }
            return sum_of(found);
        };
        // Whether no cell of the 2^bits that `cell` tells apart holds over `most` keys,
        // and all no more than `most_pairs` pairs of keys in one cell.
        auto spread = [&](uint32_t bits, uint32_t most, uint32_t most_pairs, auto cell) -> bool {
            __syncthreads();
            if (tid == 0) s_uneven = 0;
            for (uint32_t i = tid; i < (1u << bits) / 8; i += 1024)
                s_dyn[i] = make_uint4(0, 0, 0, 0);
            __syncthreads();
            uint32_t pairs = 0;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                if (NPASS == 4 && q * 1024 + tid >= samples) continue;
                const uint32_t c = cell(k[q]);
                const uint32_t was =
                    atomicAdd(&s_pair[c >> 1], 1u << (16 * (c & 1))) >> (16 * (c & 1)) & 0xffffu;
                if (was >= most) s_uneven = 1;
                pairs += was;
            }
            return sum_of(pairs) <= most_pairs && !s_uneven;
        };
        const uint32_t equal = top_equal_limit(n, NPASS == 8);
        // (32-bit keys with a digit that is the same in all are not looked at.)
        bool repeat = false;
        if (equal < samples && (NPASS == 8 || executed == NPASS)) {
            __syncthreads();  // s_uneven was read
            repeat = repeated_keys() >= equal || s_uneven;
        }
        if (top) {
            low = NPASS - 2;
            // Chunks may deviate by half of what a CTA takes over their mean.
            const float room = (float)plan.capacity / (float)(n >> top_bits) - 1.0f;
            top = !repeat && spread(top_bits, 2 * (samples >> top_bits) + 12,
                                    top_pair_limit(samples, top_bits, 0.5f * room), [&](K x) {
                                        return (uint32_t)(x >> (8 * sizeof(K) - top_bits));
                                    });
        }
        if (deep && !repeat && !top) {
            const uint32_t most = (uint32_t)(2ull * samples * plan.chunk_step / n) + 10;
            // Pairs by the hash alone, and those of prefixes of 3/4 of a CTA's items.
            const uint32_t most_pairs =
                top_pair_limit(samples, TOP_HASH_BITS) +
                (uint32_t)((3ull * plan.chunk_step / 2) * samples / 2 * samples / n);
            uint32_t passes = 0;
            for (low = NPASS; !top && low-- > 0;) {
                if (s_trivial[low]) continue;
                ++passes;
                if (passes > 4 || passes + 2 > executed) break;
                if (passes < 2) continue;
                top = spread(TOP_HASH_BITS, most, most_pairs, [&](K x) {
                    const unsigned long long h =
                        (unsigned long long)(x >> (8 * low)) * 0x9E3779B97F4A7C15ull;
                    return (uint32_t)(h >> (64 - TOP_HASH_BITS));
                });
                if (top) break;
            }
            if (tid == 0 && top) ctrl->chunk_step = plan.chunk_step;
        }
    }
    if (msd && (tid >> 8) == PASSES - 1) {
        plan.msd_off[b] = first3;
        if (b == RADIX - 1) plan.msd_off[RADIX] = n;
    }
    if (tid != 0) return;
    ctrl->dir[MSD_SLOT] = msd ? DIR_A_TO_B : DIR_SKIP;
    ctrl->small_count = msd ? RADIX : 0u;
    const uint32_t step = top ? ctrl->chunk_step : 0u;  // written above, by this thread
    ctrl->chunk_count = !top ? 0u : step != 0 ? (n + step - 1) / step : 1u << top_bits;
    ctrl->chunk_digit = low;
    bool skip[NPASS];
    for (uint32_t q = 0; q < NPASS; ++q) skip[q] = msd || s_trivial[q] || (top && q < low);
    if (!msd && !top && (executed & 1)) {
        for (uint32_t q = 0; q < NPASS; ++q)
            if (skip[q]) { skip[q] = false; break; }
    }
    uint32_t parity = 0;
    for (uint32_t q = 0; q < NPASS; ++q) {
        if (skip[q]) {
            ctrl->dir[q] = DIR_SKIP;
        } else {
            ctrl->dir[q] = parity ? DIR_B_TO_A : DIR_A_TO_B;
            parity ^= 1;
        }
    }
    ctrl->chunk_src = parity;
}

// ---------------------------------------------------------------------------
// k_chunk_bounds: the chunks of the top-digits order, once the array is sorted
// by its top digits, chunk_digit and above: off[c] = the first item of chunk c,
// off[chunk_count] = n.  Chunks by prefix: the first key with its top_bits highest
// bits equal to c or more.  Chunks by position: the first key with the prefix of
// item c * chunk_step.
// WAYS lanes search together for each bound (by prefix, in the bucket of its highest
// digit: G of that digit says where it lies; by position, in a stretch before the item
// that is made longer until it holds another prefix), reading WAYS keys at a time that
// cut what is left into WAYS + 1 parts: dependent reads are what takes the time, and 32
// ways need 3 to 4 of them where halving needs 13 to 16 (14 us for 8192 chunks of 2^24
// keys).  Many chunks take fewer ways, for the keys read.
// ---------------------------------------------------------------------------
template <typename K, int WAYS>
__global__ void __launch_bounds__(256)
k_chunk_bounds(const K* __restrict__ keys_a, const K* __restrict__ keys_b, uint32_t n,
               const Ctrl* __restrict__ ctrl, uint32_t top_bits, uint32_t key_type,
               uint32_t* __restrict__ off) {
    pdl_launch_next();
    pdl_wait();  // the scatter passes are complete
    const uint32_t chunks = ctrl->chunk_count;
    if (blockIdx.x * (256 / WAYS) >= chunks) return;
    const K* const keys = ctrl->chunk_src ? keys_b : keys_a;
    const uint32_t way = threadIdx.x % WAYS;
    const uint32_t first_lane = (threadIdx.x & 31) / WAYS * WAYS;
    // (Lanes past the last chunk search for it too, with their warp.)
    const uint32_t mine = (blockIdx.x * 256 + threadIdx.x) / WAYS;
    const uint32_t c = mine < chunks ? mine : chunks - 1;
    if (mine == 0 && way == 0) off[chunks] = n;
    const uint32_t step = ctrl->chunk_step;
    uint32_t lo, hi;  // the answer is in [lo, hi]
    K want;           // the first key not below it
    if (step == 0) {
        const uint32_t* const g = ctrl->gofs[sizeof(K) - 1];
        const uint32_t b = c >> (top_bits - RADIX_BITS);
        lo = g[b];
        hi = b + 1 < RADIX ? g[b + 1] : n;
        want = (K)c << (8 * sizeof(K) - top_bits);
    } else {
        const uint32_t shift = 8 * ctrl->chunk_digit;
        hi = c * step;
        want = key_to_ordered(keys[hi], key_type) >> shift << shift;
        uint32_t width = step;
        lo = hi > width ? hi - width : 0;
        while (lo > 0 && key_to_ordered(keys[lo], key_type) >= want) {
            width = width < (1u << 28) ? width * 8 : width;
            lo = lo > width ? lo - width : 0;
        }
    }
    while (__any_sync(0xffffffffu, lo < hi)) {
        const uint32_t part = (hi - lo) / (WAYS + 1) + 1;  // keys left of the first cut, at most
        const uint32_t at = lo + (way + 1) * part - 1;
        const bool below = at < hi && key_to_ordered(keys[at], key_type) < want;
        const uint32_t votes =
            __ballot_sync(0xffffffffu, below) >> first_lane & (0xffffffffu >> (32 - WAYS));
        const uint32_t cuts = __popc(votes);  // the first `cuts` cuts are below
        const uint32_t next = lo + cuts * part;
        hi = min(hi, next + part - 1);
        lo = min(next, hi);
    }
    if (way == 0 && mine < chunks) off[c] = lo;
}

// ---------------------------------------------------------------------------
// k_msd_plan: the plan of one stable counting-sort pass by the most
// significant digit (digit 3; Alg. 2's local MSD pass): G[3][b] = the
// exclusive prefix of H[3], copied to bucket_off[0..255] with
// bucket_off[256] = n, and the pass run (plan slot MSD_SLOT) from the input
// to the output arrays even when every key has the same digit (then it is a
// copy).  One CTA of 256 threads, thread b = bucket b.
// ---------------------------------------------------------------------------
static __global__ void __launch_bounds__(RADIX)
k_msd_plan(Ctrl* __restrict__ ctrl, uint32_t n, uint32_t* __restrict__ bucket_off) {
    __shared__ uint32_t s_warp[RADIX / 32];
    const uint32_t b = threadIdx.x, lane = b & 31, warp = b >> 5;
    const uint32_t h = ctrl->hist[PASSES - 1][b];
    uint32_t x = h;
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t off = 0;
    for (uint32_t w = 0; w < warp; ++w) off += s_warp[w];
    const uint32_t first = off + x - h;
    ctrl->gofs[PASSES - 1][b] = first;
    bucket_off[b] = first;
    if (b == 0) {
        bucket_off[RADIX] = n;
        ctrl->dir[MSD_SLOT] = DIR_A_TO_B;
    }
}

// ---------------------------------------------------------------------------
// k_hist8: the eight digit histograms of 64-bit keys (K = 64, D = 8) in one
// read of the keys, added into hist[p * 256 + b] (zeroed by the caller), via
// private columns as in k_hist4_cols: COLS = 16 (128 KiB, one CTA per SM; two lanes
// to a column) for many keys, 4 for few.  2^26 keys: 217 us with one shared histogram
// for all lanes (3.3 wavefronts an add, 8 adds a key).  Typed keys (TYPED) are counted
// by the digits of their ordered words.  Also clears the first pass's status array.
// ---------------------------------------------------------------------------
template <int COLS>
constexpr uint32_t HIST8_COL_WORDS = PASSES64 * RADIX * COLS;

template <int THREADS, int COLS, bool TYPED>
__global__ void __launch_bounds__(THREADS)
k_hist8(const unsigned long long* __restrict__ keys, uint32_t n, uint32_t* __restrict__ hist,
        uint4* __restrict__ clear, uint32_t clear_vec4, uint32_t key_type) {
    extern __shared__ uint4 s_cols4[];
    uint32_t* const s_col = reinterpret_cast<uint32_t*>(s_cols4);
    const uint32_t tid = threadIdx.x;
    pdl_launch_next();  // the plan kernel may launch; it waits for this one
    for (uint32_t i = tid; i < HIST8_COL_WORDS<COLS> / 4; i += THREADS)
        s_cols4[i] = make_uint4(0, 0, 0, 0);
    const uint32_t gtid = blockIdx.x * THREADS + tid;
    const uint32_t gsize = gridDim.x * THREADS;
    for (uint32_t i = gtid; i < clear_vec4; i += gsize) clear[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    uint32_t* const mycol = s_col + tid % COLS;
    constexpr uint32_t LOADS = 4;  // in flight per thread
    strided(gtid, LOADS * gsize, n, [&](uint32_t i, uint32_t left) {
        unsigned long long v[LOADS];
#pragma unroll
        for (uint32_t u = 0; u < LOADS; ++u)
            v[u] = u * gsize < left ? __ldcs(keys + i + u * gsize) : 0ull;
#pragma unroll
        for (uint32_t u = 0; u < LOADS; ++u) {
            if (u * gsize < left) {
                unsigned long long k = v[u];
                if (TYPED) k = key_to_ordered(k, key_type);
                const uint32_t lo = (uint32_t)k, hi = (uint32_t)(k >> 32);
#pragma unroll
                for (uint32_t p = 0; p < 4; ++p) {
                    atomicAdd(mycol + (p * RADIX + ((lo >> (8 * p)) & (RADIX - 1))) * COLS, 1u);
                    atomicAdd(mycol + ((p + 4) * RADIX + ((hi >> (8 * p)) & (RADIX - 1))) * COLS,
                              1u);
                }
            }
        }
    });
    __syncthreads();
    pdl_wait();  // the counts are zero
    for (uint32_t bin = tid; bin < PASSES64 * RADIX; bin += THREADS) {
        uint32_t c = 0;
        const uint32_t turn = bin * COLS / 32 + bin;  // 32 lanes, 32 banks
#pragma unroll
        for (uint32_t j = 0; j < COLS; ++j) c += s_col[bin * COLS + (j + turn) % COLS];
        if (c) atomicAdd(hist + bin, c);
    }
}

}  // namespace rs
