// rs_bin_sort.cuh -- k_bin_sort: one CTA sorts a whole array of up to CAP
// items on chip, by one counting step over about as many bins as there are
// items, instead of one stable counting pass per digit.
#pragma once

#include <type_traits>

#include "rs_device.cuh"

namespace rs {

// The segments of the one-warp and one-CTA sorts are listed by size, so that
// each class runs with a CTA of its own size.  Two arrays of one entry per
// segment hold the four lists, one from each end: tiny (at most warp_max items)
// from the front of `tiny`, big (more than SMALL_MID_MAX) from its back; small
// (at most SMALL_SHORT_MAX) from the front of `small`, mid from its back.
constexpr uint32_t SMALL_SHORT_MAX = 1024;
constexpr uint32_t SMALL_MID_MAX = 4096;

// Lists segment s of `size` items where it holds two or more (called by whole warps;
// one atomic per warp and list); `last` is the last entry of either array.
__device__ __forceinline__ void list_small(Ctrl* ctrl, uint32_t s, uint32_t size,
                                           uint32_t warp_max, uint32_t last, uint32_t* tiny,
                                           uint32_t* small) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t kind = size < 2                  ? 4u
                          : size <= warp_max        ? 0u
                          : size <= SMALL_SHORT_MAX ? 1u
                          : size <= SMALL_MID_MAX   ? 2u
                                                    : 3u;
    uint32_t* const counts[4] = {&ctrl->tiny_count, &ctrl->small_count, &ctrl->mid_count,
                                 &ctrl->big_count};
#pragma unroll
    for (uint32_t c = 0; c < 4; ++c) {
        const uint32_t of_kind = __ballot_sync(0xffffffffu, kind == c);
        if (of_kind == 0) continue;
        uint32_t first = 0;
        if (lane == 0) first = atomicAdd(counts[c], (uint32_t)__popc(of_kind));
        first = __shfl_sync(0xffffffffu, first, 0) + __popc(of_kind & lanemask_lt());
        if (kind != c) continue;
        if (c == 0) tiny[first] = s;
        if (c == 1) small[first] = s;
        if (c == 2) small[last - first] = s;
        if (c == 3) tiny[last - first] = s;
    }
}

// Shared-memory plan of k_bin_sort: bin words (or the counters of the digit
// passes), binned words with room for the last windows' padding, and keys (unless words
// hold them whole) and values in input order.
template <typename K, typename V, bool PAIRS, int THREADS, bool CHUNKS>
struct BinSortSmem {
    static constexpr uint32_t ITEMS = 8;  // a thread's items, and the width of a window
    static constexpr uint32_t CAP = THREADS * ITEMS;
    // Up to the power of two at or above CAP bins (chunks, whose words have no room
    // for more: 2048 or 4096), scanned by the largest power of two of threads.
    static constexpr uint32_t BIN_BITS = CAP <= 512                        ? 9
                                         : CAP <= 1024                     ? 10
                                         : CAP <= (CHUNKS ? 2560 : 2048)   ? 11
                                         : CHUNKS || CAP <= 4096           ? 12
                                                                           : 13;
    static constexpr uint32_t MAX_BINS = 1u << BIN_BITS;
    static constexpr uint32_t SCANNERS = THREADS >= 1024 ? 1024 : THREADS >= 512 ? 512
                                         : THREADS >= 256 ? 256
                                         : THREADS >= 128 ? 128 : 64;
    static constexpr uint32_t PER = MAX_BINS / SCANNERS;  // bins that a thread scans
    static_assert(PER == 4 || PER == 8 || PER == 16, "whole groups of four, swizzled");
    static constexpr uint32_t COUNTERS = (THREADS / 32) * RADIX * 4;
    static constexpr uint32_t BINS = MAX_BINS * 4 > COUNTERS ? MAX_BINS * 4 : COUNTERS;
    static constexpr uint32_t WORDS = (CAP + 2 * ITEMS) * (uint32_t)sizeof(K);
    static constexpr uint32_t KEYS = PAIRS && !CHUNKS ? CAP * (uint32_t)sizeof(K) : 0;
    static constexpr uint32_t VALS = PAIRS ? CAP * (uint32_t)sizeof(V) : 0;
    static constexpr uint32_t NEED = (THREADS + 1) * 4;  // a flag for each window
    static constexpr size_t BYTES = BINS + WORDS + KEYS + VALS + NEED;
    static_assert(BINS % 16 == 0 && WORDS % 16 == 0 && VALS % 16 == 0, "aligned parts");
};

__device__ __forceinline__ uint32_t warp_min(uint32_t x) {
    return __reduce_min_sync(0xffffffffu, x);
}
__device__ __forceinline__ unsigned long long warp_min(unsigned long long x) {
    const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32));
    const uint32_t lo =
        __reduce_min_sync(0xffffffffu, (uint32_t)(x >> 32) == hi ? (uint32_t)x : 0xffffffffu);
    return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ uint32_t leading_zeros(uint32_t x) { return __clz(x); }
__device__ __forceinline__ uint32_t leading_zeros(unsigned long long x) {
    return __clzll((long long)x);
}
__device__ __forceinline__ uint32_t high_word(uint32_t x) { return x; }
__device__ __forceinline__ uint32_t high_word(unsigned long long x) { return (uint32_t)(x >> 32); }

// Batcher's odd-even merge sort of eight words in registers.
template <typename W>
__device__ __forceinline__ void sort8(W (&w)[8]) {
    auto order = [&](int i, int j) {
        const W a = w[i], b = w[j];
        w[i] = min(a, b);
        w[j] = max(a, b);
    };
    order(0, 1), order(2, 3), order(4, 5), order(6, 7);
    order(0, 2), order(1, 3), order(4, 6), order(5, 7);
    order(1, 2), order(5, 6);
    order(0, 4), order(1, 5), order(2, 6), order(3, 7);
    order(2, 4), order(3, 5);
    order(1, 2), order(3, 4), order(5, 6);
}
// Its last steps: merges w[0..3] and w[4..7], each sorted.
template <typename W>
__device__ __forceinline__ void merge8(W (&w)[8]) {
    auto order = [&](int i, int j) {
        const W a = w[i], b = w[j];
        w[i] = min(a, b);
        w[j] = max(a, b);
    };
    order(0, 4), order(1, 5), order(2, 6), order(3, 7);
    order(2, 4), order(3, 5);
    order(1, 2), order(3, 4), order(5, 6);
}
// Sorts the eight words at p (16-byte aligned, in shared memory); HALVES: the first
// and the last four are sorted already.
template <bool HALVES, typename W>
__device__ __forceinline__ void sort_window(W* p) {
    constexpr int VECS = 8 * sizeof(W) / 16;
    union {
        uint4 v[VECS];
        W w[8];
    } u;
    // Any order (HALVES: of the halves) will do for the loads: turned so that the
    // eight lanes of a 16-byte access fall into 32 different banks (two into each,
    // for halves of 64-bit words).
    const int turn = (threadIdx.x * VECS >> 3) & (HALVES ? VECS / 2 : VECS - 1);
#pragma unroll
    for (int i = 0; i < VECS; ++i) u.v[i] = reinterpret_cast<const uint4*>(p)[i ^ turn];
    if constexpr (HALVES) merge8(u.w);
    else sort8(u.w);
#pragma unroll
    for (int i = 0; i < VECS; ++i) reinterpret_cast<uint4*>(p)[i] = u.v[i];
}

// Puts the words of the window at p (its first `left` ones) that agree but for the index
// in their `ib` lowest bits in the order of keys[index], then index.  Returns whether
// any moved.
template <typename W>
__device__ __forceinline__ bool order_ties(W* p, const W* keys, uint32_t ib, uint32_t imask,
                                           int left) {
    constexpr int VECS = 8 * sizeof(W) / 16;
    union {
        uint4 v[VECS];
        W w[8];
    } u;
#pragma unroll
    for (int i = 0; i < VECS; ++i) u.v[i] = reinterpret_cast<const uint4*>(p)[i];
    bool again = false, changed = false;
#pragma unroll
    for (int i = 0; i < 7; ++i) again |= i + 1 < left && (u.w[i] ^ u.w[i + 1]) >> ib == 0;
    if (!again) return false;
    constexpr bool CACHED = sizeof(W) == 4;  // the keys fit the registers too
    W key[CACHED ? 8 : 1];
    if constexpr (CACHED) {
#pragma unroll
        for (int i = 0; i < 8; ++i) key[i] = i < left ? keys[(uint32_t)u.w[i] & imask] : W(0);
    }
#pragma unroll 1
    while (again) {
        again = false;
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            const W a = u.w[i], b = u.w[i + 1];
            if (i + 1 < left && (a ^ b) >> ib == 0) {
                const W ka = CACHED ? key[CACHED ? i : 0] : keys[(uint32_t)a & imask];
                const W kb = CACHED ? key[CACHED ? i + 1 : 0] : keys[(uint32_t)b & imask];
                if (kb < ka || (kb == ka && b < a)) {
                    u.w[i] = b, u.w[i + 1] = a;
                    if constexpr (CACHED) key[i] = kb, key[i + 1] = ka;
                    again = changed = true;
                }
            }
        }
    }
    if (changed) {
#pragma unroll
        for (int i = 0; i < VECS; ++i) reinterpret_cast<uint4*>(p)[i] = u.v[i];
    }
    return changed;
}

// ---------------------------------------------------------------------------
// sort_in_global: one CTA sorts the m items at a (stable, in place) by counting
// passes over the 8-bit digits that differ, between a and b of the same size,
// through counters s_cnt[THREADS / 32][RADIX], s_base[RADIX] and s_hist[RADIX]; all ordered
// keys lie in [least, most].  The result is left in a, or with to_b in b.
// For the rare chunk that the top-digits order leaves too long for the chip:
// about 4 ns an item of 32 bits (one key in 0.1 % of 2^28 pairs adds 1 ms), so the plan
// counts on there being few of them, and short ones.
// ---------------------------------------------------------------------------
template <typename K, typename V, bool PAIRS, int THREADS>
__device__ __forceinline__ void sort_in_global(K* a_k, V* a_v, K* b_k, V* b_v, bool to_b,
                                               uint32_t m, uint32_t key_type, K least, K most,
                                               uint32_t* s_cnt, uint32_t* s_base,
                                               uint32_t* s_hist) {
    constexpr uint32_t WARPS = THREADS / 32, SLOTS = 4, TILE = THREADS * SLOTS;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    bool in_a = true;
#pragma unroll 1
    for (uint32_t p = 0; p < sizeof(K); ++p) {
        if (least >> (8 * p) == most >> (8 * p)) break;  // the rest is the same in all
        const K* const sk = in_a ? a_k : b_k;
        const V* const sv = in_a ? a_v : b_v;
        K* const dk = in_a ? b_k : a_k;
        V* const dv = in_a ? b_v : a_v;
        auto digit = [&](K k) {
            return (uint32_t)(key_to_ordered(k, key_type) >> (8 * p)) & (RADIX - 1);
        };
        for (uint32_t d = tid; d < RADIX; d += THREADS) s_hist[d] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < m; i += THREADS) atomicAdd(&s_hist[digit(sk[i])], 1u);
        __syncthreads();
        bool trivial = false;
        for (uint32_t d = tid; d < RADIX; d += THREADS) {
            uint32_t before = 0;
            for (uint32_t q = 0; q < d; ++q) before += s_hist[q];
            s_base[d] = before;
            trivial |= s_hist[d] == m;
        }
        if (__syncthreads_or(trivial)) continue;  // one digit only: the identity
        for (uint32_t t0 = 0; t0 < m; t0 += TILE) {
            for (uint32_t i = tid; i < WARPS * RADIX; i += THREADS) s_cnt[i] = 0;
            __syncthreads();
            K k[SLOTS];
            V v[SLOTS];
            uint32_t at[SLOTS];
#pragma unroll
            for (uint32_t j = 0; j < SLOTS; ++j) {
                const uint32_t base = t0 + (warp * SLOTS + j) * 32, i = base + lane;
                const uint32_t live = prefix_lanes(base, m);
                k[j] = i < m ? sk[i] : K(0);
                if (PAIRS && i < m) v[j] = sv[i];
                const uint32_t d = digit(k[j]);
                const uint32_t peers = match_label<RADIX_BITS>(d) & live;
                const uint32_t lead = __ffs(peers) - 1;
                uint32_t before = 0;
                if (lane == lead) before = atomicAdd(&s_cnt[warp * RADIX + d],
                                                     (uint32_t)__popc(peers));
                before = __shfl_sync(0xffffffffu, before, lead & 31u);
                at[j] = before + __popc(peers & lt);
            }
            __syncthreads();
            for (uint32_t d = tid; d < RADIX; d += THREADS) {
                uint32_t run = s_base[d];
                for (uint32_t w = 0; w < WARPS; ++w) {
                    const uint32_t c = s_cnt[w * RADIX + d];
                    s_cnt[w * RADIX + d] = run;
                    run += c;
                }
                s_base[d] = run;
            }
            __syncthreads();
#pragma unroll
            for (uint32_t j = 0; j < SLOTS; ++j) {
                if (t0 + (warp * SLOTS + j) * 32 + lane < m) {
                    const uint32_t to = at[j] + s_cnt[warp * RADIX + digit(k[j])];
                    dk[to] = k[j];
                    if (PAIRS) dv[to] = v[j];
                }
            }
            __syncthreads();  // the counters are free; the stores are visible to the CTA
        }
        in_a = !in_a;
    }
    if (in_a == to_b) {
        for (uint32_t i = tid; i < m; i += THREADS) {
            (to_b ? b_k : a_k)[i] = (to_b ? a_k : b_k)[i];
            if (PAIRS) (to_b ? b_v : a_v)[i] = (to_b ? a_v : b_v)[i];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// k_bin_sort: sorts arrays of 2 to CAP = 8 * THREADS items, one CTA per array,
// each item read from and written to global memory once.  Arrays are the segments
// listed in `list` (every `step`-th entry from it; count in *list_count), or with
// list == nullptr the segments 0, 1, ..., or with step == 0 the ranges (first item,
// items) in `list`; or with off == nullptr the single array [0, single_n).
// CHUNKS: the chunks 0, 1, ... of the top-digits order (list == nullptr), read from
// keys / vals or spare_keys / spare_vals (ctrl->chunk_src) and sorted by the digits
// from ctrl->chunk_digit on already (32-bit keys: the single_n highest bits of a chunk
// are the same); longer ones than CAP are sorted in global memory
// (sort_in_global).
//
// For an array of m items, with nb = 2^bb bins (m <= nb < 2m; chunks at most
// MAX_BINS):
//  1. The smallest and the largest key cut the range between them into nb bins of
//     the same width.  Every item adds one to its bin and keeps the count before
//     it: its place among the bin's items, in no particular order.
//  2. The exclusive prefix over bins gives every bin's first position.  Every
//     item writes its word to its bin's next position: the key, and for
//     key-value items its index below it, so that the words of a whole array
//     are in the stable order of its items.
//  3. The words are sorted up to the order inside bins, of about one item each.
//     Every thread sorts the window of eight words [8t, 8t + 8) in registers, then
//     [8t + 4, 8t + 12), and so on in turns: blocks of four words in an odd-even
//     merge, of which r rounds sort every bin that lies in r blocks.  Two or three
//     rounds of all sort most bins; the windows over longer ones take as many as the
//     longest needs (s_need).
//  4. Words leave in order, as keys, with the values their indices point to.
// Bins too long for that hold one key each (`alike`): then the bins alone are the
// order, and the index of an item inside its bin (two counting passes over (first
// position, index), none without values).  Or keys crowd: arrays then take one stable
// counting pass per 8-bit digit that differs, ranks from ballots and per-warp counters,
// items exchanged through shared memory.  An array of one key keeps its order.
//
// The word has the width of the key: the key itself without values; else the key's
// distance from the smallest, moved up until the largest has its highest bit set, with
// the index in the lowest bits.  In chunks, whose keys share as many bits as an index
// takes, that is the whole distance.  Elsewhere its lowest bits may be lost: words that
// differ in their index only are put in order by their keys, in step 4 where they are
// few (for 4096 keys that spread evenly, eight such pairs; a recount of the group by
// each of its items), or by windows in registers (order_ties).
//
// What bounds it: instruction issue (135 warp instructions per 32 pairs, 61 % of the
// issue slots) and shared-memory wavefronts (28 per 32 pairs: counting atomic, bin
// read, word write and value read at random conflicts, 3.3 each; windows 4, bins 3;
// the pipe is 60 % busy), where four digit passes take over 100; seven barriers are
// hidden by the other CTA on the SM.  Digit passes take about 130 warp instructions
// each per 32 items (61 % of the issue slots).  Ranking every item by a loop over its bin
// instead of the windows took 194 instructions, most of them in diverged loops.
// Long bins sorted by a warp each instead of by rounds of windows: 1024 segments of
// 4096 to 2^20 pairs (194 M), each key four times, 6.86 ms, now 4.07; 16 times 6.98,
// 4.30 (four scatter passes: 4.47); 2^25 keys four times each 1257 us, 513.
// Measured: chunks of 2^28 pairs 1.51 ms (2.12 by loops), of 2^28 keys 1.24; the
// 8,900 arrays of 513 to 4096 pairs among 2^15 short ones 1366 us in digit passes by
// 512-thread CTAs, 170 now; one array of 1000 keys 20.4 us against 6.6.
// ---------------------------------------------------------------------------
// The most rounds of windows, of which r sort bins of up to 4r - 3 words, and from how
// many on it is looked whether every bin holds one key.  Where 32-bit words lose bits of
// their keys, bins that long often need those put right too.  4096 segments of 256 to
// 65536 pairs with 12, 24, 32 and 48 rounds at most: 64 equal keys each 1626, 1550, 1489
// and 1371 us; ANDs of three words -, 1565, 1605 and 1758.
template <typename K, bool PAIRS, int THREADS, bool CHUNKS> struct Rounds {
    static constexpr bool LOSSY = sizeof(K) == 4 && PAIRS && !CHUNKS;
    static constexpr uint32_t MOST = !LOSSY ? 48 : THREADS <= 64 ? 12 : 24;
    static constexpr uint32_t LOOK = sizeof(K) == 4 && PAIRS ? MOST : 12;
    // That every window takes.  A third round of all windows of 64-bit words costs more
    // than to leave out those that do not need it (2^26 pairs 2.13 ms and 2.08), and of
    // 32-bit words gains a little where keys repeat a few times.
    static constexpr uint32_t ALL = sizeof(K) == 4 ? 3 : 2;
};
constexpr uint32_t FEW_ROUNDS = 3;  // up to which step 4 puts lost bits right

template <typename K, typename V, bool PAIRS, int THREADS, int MIN_BLOCKS,
          bool CHUNKS = false>
__global__ void __launch_bounds__(THREADS, MIN_BLOCKS)
k_bin_sort(K* keys, V* vals, const K* src_keys, const V* src_vals,
           const uint32_t* __restrict__ off, const uint32_t* __restrict__ list, int32_t step,
           const uint32_t* __restrict__ list_count, const Ctrl* __restrict__ ctrl,
           uint32_t single_n, uint32_t key_type, K* spare_keys, V* spare_vals) {
    using L = BinSortSmem<K, V, PAIRS, THREADS, CHUNKS>;
    constexpr bool WHOLE = !PAIRS || CHUNKS;            // words hold whole keys
    constexpr bool BY_PREFIX = CHUNKS && sizeof(K) == 4;  // 32-bit chunks all are
    using R = Rounds<K, PAIRS, THREADS, CHUNKS>;
    constexpr int ITEMS = L::ITEMS;
    constexpr uint32_t WARPS = THREADS / 32;
    constexpr uint32_t SCANNERS = L::SCANNERS;
    static_assert(WARPS <= 32 && L::CAP <= 65535, "one lane per warp total; 16-bit counts");
    pdl_launch_next();
    pdl_wait();  // the kernel before this one (planner, scatter pass) is complete
    extern __shared__ uint4 s_dyn[];
    uint32_t* const s_bin = reinterpret_cast<uint32_t*>(s_dyn);
    char* const parts = reinterpret_cast<char*>(s_dyn) + L::BINS;
    K* const s_w = reinterpret_cast<K*>(parts);
    K* const s_k = reinterpret_cast<K*>(parts + L::WORDS);
    V* const s_v = reinterpret_cast<V*>(parts + L::WORDS + L::KEYS);
    uint32_t* const s_need = reinterpret_cast<uint32_t*>(parts + L::WORDS + L::KEYS + L::VALS);
    __shared__ K s_min, s_max;
    __shared__ uint32_t s_sum[32], s_longest[32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    uint32_t count = 1;
    if (off != nullptr) {
        if (ctrl->err != 0) return;
        count = *list_count;
    }
    K sorted = 0;  // chunks: the bits of the digits they are sorted by
    if (CHUNKS && count != 0) {
        sorted = ~K(0) << (8 * ctrl->chunk_digit);
        if (ctrl->chunk_src != 0) src_keys = spare_keys, src_vals = spare_vals;
    }
    const bool typed = key_type != KEY_U32 && key_type != KEY_U64;
    if (tid == 0) s_min = ~K(0), s_max = 0;
    for (uint32_t idx = blockIdx.x; idx < count; idx += gridDim.x) {
        uint32_t lo = 0, m = single_n;
        if (off != nullptr) {
            if (!CHUNKS && step == 0) {
                lo = list[2 * idx];
                m = list[2 * idx + 1];
            } else {
                const uint32_t s = !CHUNKS && list != nullptr ? list[(ptrdiff_t)idx * step] : idx;
                lo = off[s];
                m = off[s + 1] - lo;
            }
            if (!CHUNKS && (m == 0 || m > L::CAP)) continue;
            if (CHUNKS && m == 0) continue;
            if constexpr (CHUNKS) {
                if (m > L::CAP) {
                    __syncthreads();  // the array before is done with shared memory
                    const bool b = ctrl->chunk_src != 0;
                    K* const a_k = (b ? spare_keys : keys) + lo;
                    K* const b_k = (b ? keys : spare_keys) + lo;
                    sort_in_global<K, V, PAIRS, THREADS>(
                        a_k, PAIRS ? (b ? spare_vals : vals) + lo : nullptr, b_k,
                        PAIRS ? (b ? vals : spare_vals) + lo : nullptr, b, m, key_type,
                        key_to_ordered(a_k[0], key_type) & sorted,
                        key_to_ordered(a_k[m - 1], key_type) | ~sorted, s_bin,
                        reinterpret_cast<uint32_t*>(s_w),
                        reinterpret_cast<uint32_t*>(s_w) + RADIX);
                    continue;
                }
            }
        }
        const K* const from = src_keys + lo;
        K k[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            k[j] = tid + j * THREADS < m ? from[tid + j * THREADS] : K(0);
        const uint32_t bits = m > 1 ? 32u - __clz(m - 1) : 1u;  // of an index
        const uint32_t bb = CHUNKS && bits > L::BIN_BITS ? L::BIN_BITS : bits;
        const uint32_t ib = PAIRS ? bits : 0u;
        const uint32_t nb = 1u << bb;
        const uint32_t zeroed = (nb > L::PER ? nb : L::PER) / 4;
        for (uint32_t b = tid; b < zeroed; b += THREADS)
            reinterpret_cast<uint4*>(s_bin)[b] = make_uint4(0, 0, 0, 0);
        s_need[tid] = 0;
        if (tid == 0) s_need[THREADS] = 0;
        if (typed) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) k[j] = key_to_ordered(k[j], key_type);
        }
        K least, most;
        if constexpr (CHUNKS) {
            if constexpr (BY_PREFIX) {  // the keys share their single_n highest bits
                const K low_bits = ~K(0) >> single_n;
                least = key_to_ordered(from[0], key_type) & ~low_bits;
                most = least | low_bits;
            } else {  // the ends' sorted digits say
                least = key_to_ordered(from[0], key_type) & sorted;
                most = key_to_ordered(from[m - 1], key_type) | ~sorted;
            }
            __syncthreads();  // the bins are zero; the array before is done with the rest
        } else {
            K lo_k = ~K(0), not_hi = ~K(0);
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                if (tid + j * THREADS < m) {
                    lo_k = min(lo_k, k[j]);
                    not_hi = min(not_hi, ~k[j]);
                }
            }
            lo_k = warp_min(lo_k);
            not_hi = warp_min(not_hi);
            __syncthreads();  // s_min, s_max and the bins are set; as above
            if (lane == 0) {
                atomicMin(&s_min, lo_k);
                atomicMax(&s_max, ~not_hi);
            }
            __syncthreads();
            least = s_min;
            most = s_max;
            if (least == most) {  // one key: the items stay in their order
                __syncthreads();  // all have read it
                if (tid == 0) s_min = ~K(0), s_max = 0;  // for the next array
                if (src_keys == keys) continue;
#pragma unroll 1
                for (uint32_t i = tid; i < m; i += THREADS) {
                    keys[lo + i] = from[i];
                    if (PAIRS) vals[lo + i] = src_vals[lo + i];
                }
                continue;
            }
        }
        const K range = (most - least) | 1;
        if (PAIRS) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m)
                    cp_async_elem(s_v + tid + j * THREADS, src_vals + lo + tid + j * THREADS);
        }
        const uint32_t top = BY_PREFIX ? single_n : leading_zeros(range);  // bits of 0 in all
        // Bins: distance * scale / 2^32, of the (high words of the) distances moved up
        // by `top`; scale is nb * 2^32 / (range + 1), or up to 2e-6 of it less (a
        // quotient of floats, kept below the exact one, so that every bin is below nb).
        uint32_t scale = nb;
        if constexpr (!BY_PREFIX)
            scale = (uint32_t)(__fdividef((float)nb * 4294967296.0f,
                                          (float)high_word((K)(range << top))) * 0.999999f);
        // Scanning thread t scans the PER consecutive bins from t * PER on, four at a
        // time; their groups of four are swizzled so that the eight lanes of a 16-byte
        // access fall into 32 different banks.
        constexpr uint32_t PER = L::PER, SWIZZLE = (PER / 4 - 1) << 2;
        auto swizzled = [](uint32_t b) { return b ^ ((b >> 3) & SWIZZLE); };
        auto bin_of = [&](K x) {
            return swizzled(BY_PREFIX ? high_word((K)(x << top)) >> (32 - bb)
                                      : __umulhi(high_word((K)((x - least) << top)), scale));
        };

        // ---- 1. count, keeping each item's place among its bin's items ------
        uint32_t at[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (tid + j * THREADS < m) at[j] = atomicAdd(&s_bin[bin_of(k[j])], 1u);
        __syncthreads();

        // ---- 2. exclusive prefix over the bins ------------------------------
        // Bins become first positions; `longest` is the longest bin's length.
        uint32_t longest = 0;
        {
            const bool scans = tid < SCANNERS && tid * PER < nb;
            uint32_t c[PER];
            uint32_t sum = 0;
            constexpr uint32_t VECS = PER / 4;
            uint4* const vec = reinterpret_cast<uint4*>(s_bin) + tid * VECS;
            const uint32_t turn = (tid * PER >> 5) & (VECS - 1);  // the swizzle of its groups
#pragma unroll
            for (uint32_t g = 0; g < VECS; ++g) {
                const uint4 x = scans ? vec[g ^ turn] : make_uint4(0, 0, 0, 0);
                c[4 * g] = x.x, c[4 * g + 1] = x.y, c[4 * g + 2] = x.z, c[4 * g + 3] = x.w;
            }
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                sum += c[q];
                longest = max(longest, c[q]);
            }
            uint32_t x = sum;
#pragma unroll
            for (uint32_t o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            longest = __reduce_max_sync(0xffffffffu, longest);
            if (lane == 31) {
                s_sum[warp] = x;
                s_longest[warp] = longest;
            }
            __syncthreads();
            const uint32_t before = lane < warp ? s_sum[lane] : 0u;
            longest = __reduce_max_sync(0xffffffffu, lane < WARPS ? s_longest[lane] : 0u);
            uint32_t run = __reduce_add_sync(0xffffffffu, before) + x - sum;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                const uint32_t e = run;
                run += c[q];
                c[q] = e;
            }
#pragma unroll
            for (uint32_t g = 0; g < VECS; ++g)
                if (scans)
                    vec[g ^ turn] = make_uint4(c[4 * g], c[4 * g + 1], c[4 * g + 2], c[4 * g + 3]);
        }
        if (tid == 0) s_min = ~K(0), s_max = 0;  // for the next array
        __syncthreads();

        // Windows of words, in as many rounds as the longest bin takes; or where it is too
        // long for that, and every bin holds one key (`alike`), none for keys only.
        // (Chunks whose words would not hold whole keys take the digit passes too: none
        // by prefix; by position, where the keys are sparse.)
        uint32_t rounds = (longest + 6) / 4;
        bool windowed = !CHUNKS || ib <= top, alike = false;
        if (rounds > R::LOOK) {
            K* const first_of = s_w;  // a key of every bin, at the bin's first position
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m) first_of[s_bin[bin_of(k[j])]] = k[j];
            __syncthreads();
            bool same = true;
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m) same &= first_of[s_bin[bin_of(k[j])]] == k[j];
            alike = __syncthreads_and(same);
            if (alike || rounds > R::MOST) windowed = alike && !PAIRS;
            if (alike) rounds = 0;
        }
        if (windowed) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m) {
                    const uint32_t i = tid + j * THREADS;
                    K w = k[j];
                    if (PAIRS && CHUNKS) w = ((BY_PREFIX ? w : w - least) << top) | (K)i;
                    if (PAIRS && !CHUNKS) w = ((w - least) << top >> ib << ib) | (K)i;
                    const uint32_t first = s_bin[bin_of(k[j])];
                    s_w[first + at[j]] = w;
                    if (!WHOLE) s_k[i] = k[j];
                    if (at[j] >= 4 * R::ALL - 3) {  // in a longer bin: its windows
                        s_need[(first + at[j]) / 8] = 1;
                        if (at[j] == 4 * R::ALL - 3)
                            for (uint32_t x = first / 8; x < (first + at[j]) / 8; ++x)
                                s_need[x] = 1;
                    }
                }
            // Padding above every word, to the end of the last window.
            const uint32_t windows = (m + 7) / 8;
            const uint32_t imask = (1u << bits) - 1;
            if (tid < 8 * windows + 8 - m) s_w[m + tid] = ~K(0);
            __syncthreads();
            // ---- 3. the order inside bins ----------------------------------
            if (rounds != 0) {
                if (tid < windows) sort_window<false>(s_w + 8 * tid);
#pragma unroll 1
                for (uint32_t r = 1; r < rounds; ++r) {
                    __syncthreads();
                    if (tid < windows &&
                        (r < R::ALL || s_need[tid] != 0 || ((r & 1) && s_need[tid + 1] != 0)))
                        sort_window<true>(s_w + 8 * tid + 4 * (r & 1));
                }
                if constexpr (!WHOLE) {
                    // Words next to each other may differ in their index only because the
                    // key's last bits did not fit: those are put in order by their keys,
                    // until no window of either row has changed.  (Few of them: in step 4.)
                    uint32_t done = rounds > FEW_ROUNDS ? 0 : 2;
#pragma unroll 1
                    for (uint32_t r = 0; done < 2; ++r) {
                        __syncthreads();
                        const uint32_t at_ = 8 * tid + 4 * (r & 1);
                        const bool changed =
                            tid < windows &&
                            order_ties(s_w + at_, s_k, ib, imask, (int)m - (int)at_);
                        done = __syncthreads_or(changed) ? 0 : done + 1;
                    }
                }
            }
            if (PAIRS) cp_async_wait_all();
            __syncthreads();
            // ---- 4. stored in order -----------------------------------------
            uint32_t tied = 0;  // items whose word differs from a neighbour's in the index only
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t at_ = tid + j * THREADS;
                if (at_ < m) {
                    const K w = s_w[at_];
                    if (!WHOLE && rounds <= FEW_ROUNDS &&
                        ((at_ > 0 && (s_w[at_ - 1] ^ w) >> ib == 0) ||
                         (at_ + 1 < m && (s_w[at_ + 1] ^ w) >> ib == 0))) {
                        tied |= 1u << j;
                        continue;
                    }
                    const uint32_t i = (uint32_t)w & imask;
                    K key;
                    if constexpr (WHOLE) key = PAIRS ? (K)(w >> top) + least : w;
                    else key = s_k[i];
                    if (typed) key = key_from_ordered(key, key_type);
                    keys[lo + at_] = key;
                    if (PAIRS) vals[lo + at_] = s_v[i];
                }
            }
            // Those find their places among each other by their keys.
#pragma unroll 1
            for (; !WHOLE && tied != 0; tied &= tied - 1) {
                const uint32_t at_ = tid + (__ffs(tied) - 1) * THREADS;
                const K w = s_w[at_];
                const uint32_t i = (uint32_t)w & imask;
                K key = s_k[i];
                uint32_t to = at_, last = at_;
#pragma unroll 1
                while (to > 0 && (s_w[to - 1] ^ w) >> ib == 0) --to;
#pragma unroll 1
                while (last + 1 < m && (s_w[last + 1] ^ w) >> ib == 0) ++last;
#pragma unroll 1
                for (uint32_t q = to; q <= last; ++q) {
                    const uint32_t o = (uint32_t)s_w[q] & imask;
                    const K ok = s_k[o];
                    to += ok < key || (ok == key && o < i) ? 1u : 0u;
                }
                if (typed) key = key_from_ordered(key, key_type);
                keys[lo + to] = key;
                if (PAIRS) vals[lo + to] = s_v[i];
            }
        } else {
            // ---- digit passes ------------------------------------------------
            // Warp w holds the items [w * 32 * ipt, (w + 1) * 32 * ipt), slot by
            // slot: (warp, slot, lane) order is the input order.  Items stay in
            // registers; a pass moves them to their new slots through shared
            // memory.
            const uint32_t ipt = (m + THREADS - 1) / THREADS;
            const uint32_t me = warp * 32 * ipt + lane;
            const uint32_t left = m > me ? (m - me + 31) / 32 : 0u;
            const uint32_t mine = left < ipt ? left : ipt;
            const uint32_t lt = lanemask_lt();
            uint32_t* const row = s_bin + warp * RADIX;
            V v[PAIRS ? ITEMS : 1];
            // alike: words of the bin's first position above the item's index.
            constexpr uint32_t INDEX_BITS = 13, INDEX_MASK = (1u << INDEX_BITS) - 1;
            static_assert(L::CAP <= 1u << INDEX_BITS, "positions and indices fit");
            const bool by_bin = PAIRS && alike;
            if (PAIRS) cp_async_wait_all();
            __syncthreads();
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                if (j < mine) {
                    k[j] = key_to_ordered(from[me + j * 32], key_type);
                    if (by_bin) k[j] = (K)s_bin[bin_of(k[j])] << INDEX_BITS | (me + j * 32);
                    else if (PAIRS) v[j] = s_v[me + j * 32];
                }
            }
            __syncthreads();  // the bins are read: counters take their place
#pragma unroll 1
            for (uint32_t shift = by_bin ? INDEX_BITS : 0;
                 by_bin ? shift < INDEX_BITS + bits
                        : shift < 8 * sizeof(K) && least >> shift != most >> shift;
                 shift += RADIX_BITS) {
                for (uint32_t b = lane; b < RADIX; b += 32) row[b] = 0;
                __syncwarp();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < ipt) {
                        const uint32_t d = (uint32_t)(k[j] >> shift) & (RADIX - 1);
                        const uint32_t live = prefix_lanes(me - lane + j * 32, m);
                        const uint32_t peers = match_label<RADIX_BITS>(d) & live;
                        const uint32_t lead = __ffs(peers) - 1;
                        uint32_t before = 0;
                        if (lane == lead) before = atomicAdd(&row[d], (uint32_t)__popc(peers));
                        before = __shfl_sync(0xffffffffu, before, lead & 31u);
                        at[j] = before + __popc(peers & lt);
                    }
                }
                __syncthreads();
                // Thread t turns the counts of its consecutive digits into
                // every warp's first position of the digit.
                constexpr uint32_t DIGITS = RADIX > THREADS ? RADIX / THREADS : 1;
                uint32_t c[DIGITS], sum = 0;
                bool trivial = false;
#pragma unroll
                for (uint32_t q = 0; q < DIGITS; ++q) {
                    c[q] = 0;
                    const uint32_t d = tid * DIGITS + q;
                    if (d < RADIX)
                        for (uint32_t w = 0; w < WARPS; ++w) c[q] += s_bin[w * RADIX + d];
                    trivial |= c[q] == m;
                    sum += c[q];
                }
                if (__syncthreads_or(trivial)) continue;  // one digit only: the identity
                uint32_t x = sum;
#pragma unroll
                for (uint32_t o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (lane == 31) s_sum[warp] = x;
                __syncthreads();
                const uint32_t before = lane < warp ? s_sum[lane] : 0u;
                uint32_t run = __reduce_add_sync(0xffffffffu, before) + x - sum;
#pragma unroll
                for (uint32_t q = 0; q < DIGITS; ++q) {
                    const uint32_t d = tid * DIGITS + q;
                    if (d < RADIX) {
                        uint32_t r = run;
                        constexpr uint32_t BATCH = WARPS < 6 ? WARPS : 6;  // reads in flight
                        for (uint32_t w0 = 0; w0 < WARPS; w0 += BATCH) {
                            uint32_t t[BATCH];
#pragma unroll
                            for (uint32_t w = 0; w < BATCH; ++w)
                                t[w] = w0 + w < WARPS ? s_bin[(w0 + w) * RADIX + d] : 0u;
#pragma unroll
                            for (uint32_t w = 0; w < BATCH; ++w) {
                                if (w0 + w < WARPS) s_bin[(w0 + w) * RADIX + d] = r;
                                r += t[w];
                            }
                        }
                    }
                    run += c[q];
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < mine) {
                        at[j] += row[(uint32_t)(k[j] >> shift) & (RADIX - 1)];
                        s_w[at[j]] = k[j];
                        if (PAIRS && !by_bin) s_v[at[j]] = v[j];
                    }
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < mine) {
                        k[j] = s_w[me + j * 32];
                        if (PAIRS && !by_bin) v[j] = s_v[me + j * 32];
                    }
                }
                __syncthreads();
            }
            if (by_bin) {
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < mine) {
                        const uint32_t i = (uint32_t)k[j] & INDEX_MASK;
                        k[j] = key_to_ordered(from[i], key_type);
                        v[PAIRS ? j : 0] = s_v[i];
                    }
                }
                __syncthreads();  // every key is read before any is stored
            }
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t i = me + j * 32;
                if (j < mine) {
                    keys[lo + i] = key_from_ordered(k[j], key_type);
                    if (PAIRS) vals[lo + i] = v[j];
                }
            }
        }
    }
}

}  // namespace rs
