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

// Lists segment s of `size` items (more than warp_max, or tiny); `last` is the
// last entry of either array.
__device__ __forceinline__ void list_small(Ctrl* ctrl, uint32_t s, uint32_t size,
                                           uint32_t warp_max, uint32_t last, uint32_t* tiny,
                                           uint32_t* small) {
    if (size <= warp_max) tiny[atomicAdd(&ctrl->tiny_count, 1u)] = s;
    else if (size <= SMALL_SHORT_MAX) small[atomicAdd(&ctrl->small_count, 1u)] = s;
    else if (size <= SMALL_MID_MAX) small[last - atomicAdd(&ctrl->mid_count, 1u)] = s;
    else tiny[last - atomicAdd(&ctrl->big_count, 1u)] = s;
}

// Shared-memory plan of k_bin_sort: bin words (or the counters of the digit
// passes), binned words with room for the last windows' padding, values in input
// order, and the list of bins that the windows do not cover.
template <typename K, typename V, typename W, bool PAIRS, int THREADS, bool CHUNKS>
struct BinSortSmem {
    static constexpr uint32_t ITEMS = 8;  // a thread's items, and the width of a window
    static constexpr uint32_t CAP = THREADS * ITEMS;
    // Up to the power of two at or above CAP bins (chunks, whose words have no room
    // for more: 2048 or 4096), scanned by the largest power of two of threads.
    static constexpr uint32_t BIN_BITS =
        CAP <= 1024 ? 10 : CAP <= (CHUNKS ? 2560 : 2048) ? 11 : CHUNKS || CAP <= 4096 ? 12 : 13;
    static constexpr uint32_t MAX_BINS = 1u << BIN_BITS;
    static constexpr uint32_t SCANNERS = THREADS >= 1024 ? 1024 : THREADS >= 512 ? 512
                                         : THREADS >= 256 ? 256 : 128;
    static constexpr uint32_t COUNTERS = (THREADS / 32) * RADIX * 4;
    static constexpr uint32_t BINS = MAX_BINS * 4 > COUNTERS ? MAX_BINS * 4 : COUNTERS;
    static constexpr uint32_t WORDS = (CAP + 2 * ITEMS) * (uint32_t)sizeof(W);
    static constexpr uint32_t VALS = PAIRS ? CAP * (uint32_t)sizeof(V) : 0;
    static constexpr uint32_t BIG = (CAP / 6 + 1) * 4;
    static constexpr size_t BYTES = BINS + WORDS + VALS + BIG;
    static_assert(BINS % 16 == 0 && WORDS % 16 == 0 && VALS % 16 == 0, "aligned parts");
};

__device__ __forceinline__ uint32_t warp_or(uint32_t x) {
    return __reduce_or_sync(0xffffffffu, x);
}
__device__ __forceinline__ unsigned long long warp_or(unsigned long long x) {
    return ((unsigned long long)__reduce_or_sync(0xffffffffu, (uint32_t)(x >> 32)) << 32) |
           __reduce_or_sync(0xffffffffu, (uint32_t)x);
}
__device__ __forceinline__ uint32_t significant_bits(uint32_t x) { return 32u - __clz(x); }
__device__ __forceinline__ uint32_t significant_bits(unsigned long long x) {
    return 64u - __clzll((long long)x);
}

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
// Sorts the eight words at p (16-byte aligned, in shared memory).
template <typename W>
__device__ __forceinline__ void sort_window(W* p) {
    constexpr int VECS = 8 * sizeof(W) / 16;
    union {
        uint4 v[VECS];
        W w[8];
    } u;
    // Any order will do for the loads: turned so that the eight lanes of a
    // 16-byte access fall into 32 different banks.
    const int turn = (threadIdx.x * VECS >> 3) & (VECS - 1);
#pragma unroll
    for (int i = 0; i < VECS; ++i) u.v[i] = reinterpret_cast<const uint4*>(p)[i ^ turn];
    sort8(u.w);
#pragma unroll
    for (int i = 0; i < VECS; ++i) reinterpret_cast<uint4*>(p)[i] = u.v[i];
}

// ---------------------------------------------------------------------------
// sort_in_global: one CTA sorts the m items at a (stable, in place) by counting
// passes over the 8-bit digits that differ, between a and b of the same size,
// through counters s_cnt[THREADS / 32][RADIX], s_base[RADIX] and s_hist[RADIX].
// For the rare chunk that the top-digits order leaves too long for the chip:
// about 1 item per ns, so it counts on there being few of them.
// ---------------------------------------------------------------------------
template <typename K, typename V, bool PAIRS, int THREADS>
__device__ __forceinline__ void sort_in_global(K* a_k, V* a_v, K* b_k, V* b_v, uint32_t m,
                                            uint32_t key_type, uint32_t* s_cnt, uint32_t* s_base,
                                            uint32_t* s_hist) {
    constexpr uint32_t WARPS = THREADS / 32, SLOTS = 4, TILE = THREADS * SLOTS;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    bool in_a = true;
    for (uint32_t p = 0; p < sizeof(K); ++p) {
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
    if (!in_a) {
        for (uint32_t i = tid; i < m; i += THREADS) {
            a_k[i] = b_k[i];
            if (PAIRS) a_v[i] = b_v[i];
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// k_bin_sort: sorts arrays of 2 to CAP = 8 * THREADS items, one CTA per array,
// each item read from and written to global memory once.  Arrays are the segments
// listed in `list` (every `step`-th entry from it; count in *list_count), or with
// list == nullptr those of the segments 0, 1, ... that hold more than single_n
// items and at most CAP; or with off == nullptr the single array [0, single_n).
// CHUNKS: the segments 0, 1, ... (list == nullptr), sorted in place; longer ones
// than CAP in global memory, with the other buffer at spare_keys / spare_vals
// (sort_in_global); their keys share the single_n highest bits.
//
// For an array of m items, with nb = 2^bb bins (m <= nb < 2m; chunks at most
// MAX_BINS):
//  1. The keys' bits that differ (an OR over the array) say where the bb
//     highest of them lie; those are the item's bin.  Every item adds one to
//     its bin and keeps the count before it: its place among the bin's items,
//     in no particular order.
//  2. The exclusive prefix over bins gives every bin's first position.  Every
//     item writes its word to its bin's next position: the key, and for
//     key-value items its index below it, so that the words of a whole array
//     are in the stable order of its items.
//  3. The words are sorted up to the order inside bins, of about one item each.
//     Every thread sorts the window of eight words [8t, 8t + 8) in registers, then
//     [8t + 4, 8t + 12): every bin of at most five lies within one of them.
//     Longer bins are listed in step 2 and sorted before, one warp per bin, by
//     counting the smaller words.
//  4. Words leave in order, as keys, with the values their indices point to.
// Arrays whose keys crowd into few bins (the work of the listed bins is known
// after step 2; the line is at one comparison by a warp for each item, and at
// WARP_BIN_MAX items in a bin) take one
// stable counting pass per 8-bit digit that differs instead: ranks from ballots
// and per-warp counters, items exchanged through shared memory.
//
// The word: W = K without values; 64-bit words hold any 32-bit key and its index;
// 32-bit words (64-bit for 64-bit keys) hold the index and the low bits of the
// key where the others are the same in the whole array, as in chunks.
//
// What bounds it: instruction issue (135 warp instructions per 32 pairs, 61 % of the
// issue slots) and shared-memory wavefronts (28 per 32 pairs: counting atomic, bin
// read, word write and value read at random conflicts, 3.3 each; windows 4, bins 3;
// the pipe is 60 % busy), where four digit passes take over 100; seven barriers are
// hidden by the other CTA on the SM.  Ranking every item by a loop over its bin
// instead of the windows took 194 instructions, most of them in diverged loops.
// Measured: chunks of 2^28 pairs 1.51 ms (2.12 by loops), of 2^28 keys 1.24; the
// 8,900 arrays of 513 to 4096 pairs among 2^15 short ones 1366 us in digit passes by
// 512-thread CTAs, 170 now; one array of 1000 keys 20.4 us against 6.6.
// ---------------------------------------------------------------------------
constexpr uint32_t WINDOW_BIN_MAX = 5;  // the longest bin that the windows sort
constexpr uint32_t WARP_BIN_MAX = 128;  // the longest bin that a warp sorts

// One warp sorts the c <= WARP_BIN_MAX words of a bin: every word goes to the
// number of words below it (TIES: equal ones in their present order).
template <typename W, bool TIES>
__device__ __forceinline__ void sort_bin(W* bin, uint32_t c, uint32_t lane) {
    constexpr uint32_t R = WARP_BIN_MAX / 32;
    W w[R];
    uint32_t pos[R];
#pragma unroll
    for (uint32_t r = 0; r < R; ++r) {
        w[r] = bin[r * 32 + lane < c ? r * 32 + lane : 0];
        pos[r] = 0;
    }
    for (uint32_t q = 0; q < c; ++q) {
        const W o = bin[q];
#pragma unroll
        for (uint32_t r = 0; r < R; ++r)
            if (r * 32 < c)
                pos[r] += o < w[r] || (TIES && o == w[r] && q < r * 32 + lane) ? 1u : 0u;
    }
    __syncwarp();
#pragma unroll
    for (uint32_t r = 0; r < R; ++r)
        if (r * 32 + lane < c) bin[pos[r]] = w[r];
}

template <typename K, typename V, typename W, bool PAIRS, int THREADS, int MIN_BLOCKS,
          bool CHUNKS = false>
__global__ void __launch_bounds__(THREADS, MIN_BLOCKS)
k_bin_sort(K* keys, V* vals, const K* src_keys, const V* src_vals,
           const uint32_t* __restrict__ off, const uint32_t* __restrict__ list, int32_t step,
           const uint32_t* __restrict__ list_count, const Ctrl* __restrict__ ctrl,
           uint32_t single_n, uint32_t key_type, K* spare_keys, V* spare_vals) {
    using L = BinSortSmem<K, V, W, PAIRS, THREADS, CHUNKS>;
    constexpr int ITEMS = L::ITEMS;
    constexpr uint32_t WARPS = THREADS / 32;
    constexpr uint32_t SCANNERS = L::SCANNERS;
    static_assert(WARPS <= 32 && L::CAP <= 65535, "one lane per warp total; 16-bit counts");
    static_assert(sizeof(W) >= sizeof(K), "a word holds a key");
    pdl_launch_next();
    pdl_wait();  // the kernel before this one (planner, scatter pass) is complete
    extern __shared__ uint4 s_dyn[];
    uint32_t* const s_bin = reinterpret_cast<uint32_t*>(s_dyn);
    W* const s_w = reinterpret_cast<W*>(reinterpret_cast<char*>(s_dyn) + L::BINS);
    V* const s_v = reinterpret_cast<V*>(reinterpret_cast<char*>(s_dyn) + L::BINS + L::WORDS);
    uint32_t* const s_big = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(s_dyn) + L::BINS +
                                                        L::WORDS + L::VALS);
    __shared__ K s_or;
    __shared__ uint32_t s_sum[32], s_work[32];
    __shared__ uint32_t s_bigs;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    uint32_t count = 1;
    if (off != nullptr) {
        if (ctrl->err != 0) return;
        count = *list_count;
    }
    const bool typed = key_type != KEY_U32 && key_type != KEY_U64;
    if (tid == 0) s_or = 0, s_bigs = 0;
    for (uint32_t idx = blockIdx.x; idx < count; idx += gridDim.x) {
        uint32_t lo = 0, m = single_n;
        if (off != nullptr) {
            const uint32_t s = !CHUNKS && list != nullptr ? list[(ptrdiff_t)idx * step] : idx;
            lo = off[s];
            m = off[s + 1] - lo;
            if (!CHUNKS && list == nullptr && (m <= single_n || m > L::CAP)) continue;
            if (CHUNKS && m < 2) continue;
            if constexpr (CHUNKS) {
                if (m > L::CAP) {
                    __syncthreads();  // the array before is done with shared memory
                    sort_in_global<K, V, PAIRS, THREADS>(
                        keys + lo, PAIRS ? vals + lo : nullptr, spare_keys + lo,
                        PAIRS ? spare_vals + lo : nullptr, m, key_type, s_bin,
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
        for (uint32_t b = tid; b < (nb + 3) / 4; b += THREADS)
            reinterpret_cast<uint4*>(s_bin)[b] = make_uint4(0, 0, 0, 0);
        const K first = key_to_ordered(from[0], key_type);
        K varying = ~K(0) >> (CHUNKS ? single_n : 0u), diff = 0;
        if (typed) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) k[j] = key_to_ordered(k[j], key_type);
        }
        if (!CHUNKS) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m) diff |= k[j] ^ first;
        }
        __syncthreads();  // the bins are zero; the array before is done with the words and values
        if (PAIRS) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m)
                    cp_async_elem(s_v + tid + j * THREADS, src_vals + lo + tid + j * THREADS);
        }
        if (!CHUNKS) {
            diff = warp_or(diff);
            if (lane == 0 && diff != 0) atomicOr(&s_or, diff);
            __syncthreads();
            varying = s_or;
        }
        const uint32_t sig = significant_bits(varying);
        const uint32_t shift = sig > bb ? sig - bb : 0u;
        // Scanning thread t scans the `per` consecutive bins from t * per on,
        // four at a time; their groups of four are swizzled so that the eight
        // lanes of a 16-byte access fall into 32 different banks.
        const uint32_t per = nb > SCANNERS ? nb / SCANNERS : 1u;  // 1, 2, 4, 8 or 16
        const uint32_t swizzle = per > 4 ? (per / 4 - 1) << 2 : 0u;
        auto bin_of = [&](K x) {
            const uint32_t b = (uint32_t)(x >> shift) & (nb - 1);
            return b ^ ((b >> 3) & swizzle);
        };

        // ---- 1. count, keeping each item's place among its bin's items ------
        uint32_t at[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (tid + j * THREADS < m) at[j] = atomicAdd(&s_bin[bin_of(k[j])], 1u);
        __syncthreads();

        // ---- 2. exclusive prefix over the bins ------------------------------
        // Bins become first positions.  Returns the work of the long bins, which
        // are listed as (first position, count << 16).
        auto scan_bins = [&](auto per_) {
            constexpr uint32_t PER = decltype(per_)::value;
            const bool scans = tid < SCANNERS && tid * PER < nb;
            uint32_t c[PER];
            uint32_t sum = 0, work = 0;
            constexpr uint32_t VECS = PER >= 4 ? PER / 4 : 1;
            uint4* const vec = reinterpret_cast<uint4*>(s_bin) + tid * VECS;
            const uint32_t turn = (tid * PER >> 5) & (VECS - 1);  // the swizzle of its groups
            if constexpr (PER >= 4) {
#pragma unroll
                for (uint32_t g = 0; g < VECS; ++g) {
                    const uint4 x = scans ? vec[g ^ turn] : make_uint4(0, 0, 0, 0);
                    c[4 * g] = x.x, c[4 * g + 1] = x.y, c[4 * g + 2] = x.z, c[4 * g + 3] = x.w;
                }
            } else {
#pragma unroll
                for (uint32_t q = 0; q < PER; ++q) c[q] = scans ? s_bin[tid * PER + q] : 0u;
            }
            uint32_t longest = 0;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                sum += c[q];
                longest = max(longest, c[q]);
            }
            if (longest > WINDOW_BIN_MAX) {
#pragma unroll
                for (uint32_t q = 0; q < PER; ++q)
                    if (c[q] > WINDOW_BIN_MAX)
                        work += c[q] <= WARP_BIN_MAX ? (c[q] + 31) / 32 * c[q] : L::CAP + 1;
            }
            uint32_t x = sum;
#pragma unroll
            for (uint32_t o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            const uint32_t warp_work = __reduce_add_sync(0xffffffffu, work);
            if (lane == 31) {
                s_sum[warp] = x;
                s_work[warp] = warp_work;
            }
            __syncthreads();
            const uint32_t before = lane < warp ? s_sum[lane] : 0u;
            const uint32_t all = lane < WARPS ? s_work[lane] : 0u;
            uint32_t run = __reduce_add_sync(0xffffffffu, before) + x - sum;
            if (longest > WINDOW_BIN_MAX) {
                uint32_t at_bin = run;
#pragma unroll
                for (uint32_t q = 0; q < PER; ++q) {
                    if (c[q] > WINDOW_BIN_MAX)
                        s_big[atomicAdd(&s_bigs, 1u)] = at_bin | (c[q] << 16);
                    at_bin += c[q];
                }
            }
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                const uint32_t e = run;
                run += c[q];
                c[q] = e;
            }
            if constexpr (PER >= 4) {
#pragma unroll
                for (uint32_t g = 0; g < VECS; ++g)
                    if (scans) vec[g ^ turn] = make_uint4(c[4 * g], c[4 * g + 1], c[4 * g + 2],
                                                          c[4 * g + 3]);
            } else {
#pragma unroll
                for (uint32_t q = 0; q < PER; ++q)
                    if (scans) s_bin[tid * PER + q] = c[q];
            }
            return __reduce_add_sync(0xffffffffu, all);
        };
        uint32_t work;
        constexpr uint32_t MAX_PER = L::MAX_BINS / SCANNERS;
        static_assert(MAX_PER >= 4 && MAX_PER <= 16, "see the dispatch below");
        if (per == 1) work = scan_bins(std::integral_constant<uint32_t, 1>{});
        else if (per == 2) work = scan_bins(std::integral_constant<uint32_t, 2>{});
        else if (per == 4 || MAX_PER == 4) work = scan_bins(std::integral_constant<uint32_t, 4>{});
        else if (per == 8 || MAX_PER == 8) work = scan_bins(std::integral_constant<uint32_t, 8>{});
        else work = scan_bins(std::integral_constant<uint32_t, MAX_PER>{});
        if (tid == 0) s_or = 0;  // for the next array
        __syncthreads();
        const uint32_t bigs = s_bigs;

        // Words that the word type cannot hold in order (see above) take the
        // digit passes too; the callers' choices of W leave none.
        if (work <= m && sig + ib <= 8 * sizeof(W)) {
#pragma unroll
            for (int j = 0; j < ITEMS; ++j)
                if (tid + j * THREADS < m)
                    s_w[s_bin[bin_of(k[j])] + at[j]] =
                        ((W)k[j] << ib) | (PAIRS ? (W)(tid + j * THREADS) : W(0));
            // Padding above every word, to the end of the last window.
            const uint32_t windows = (m + 7) / 8;
            if (tid < 8 * windows + 8 - m) s_w[m + tid] = ~W(0);
            __syncthreads();
            // ---- 3. the order inside bins ----------------------------------
            if (bigs != 0) {
                for (uint32_t g = warp; g < bigs; g += WARPS) {
                    sort_bin<W, !PAIRS>(s_w + (s_big[g] & 0xffffu), s_big[g] >> 16, lane);
                }
                if (tid == 0) s_bigs = 0;  // for the next array (read above, before a barrier)
                __syncthreads();
            }
            if (tid < windows) sort_window(s_w + 8 * tid);
            __syncthreads();
            if (tid < windows) sort_window(s_w + 8 * tid + 4);
            if (PAIRS) cp_async_wait_all();
            __syncthreads();
            // ---- 4. stored in order -----------------------------------------
            const K high = PAIRS && sizeof(W) == sizeof(K) ? first & ~(~K(0) >> ib) : K(0);
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t i = tid + j * THREADS;
                if (i < m) {
                    const W w = s_w[i];
                    K key = (K)(w >> ib) | high;
                    if (typed) key = key_from_ordered(key, key_type);
                    keys[lo + i] = key;
                    if (PAIRS) vals[lo + i] = s_v[(uint32_t)w & ((1u << bits) - 1)];
                }
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
            K* const s_k = reinterpret_cast<K*>(s_w);
            V v[PAIRS ? ITEMS : 1];
            if (PAIRS) cp_async_wait_all();
            __syncthreads();
            if (tid == 0) s_bigs = 0;  // for the next array
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                if (j < mine) {
                    k[j] = key_to_ordered(from[me + j * 32], key_type);
                    if (PAIRS) v[j] = s_v[me + j * 32];
                }
            }
            for (uint32_t p = 0; p < sizeof(K); ++p) {
                if (((varying >> (8 * p)) & (RADIX - 1)) == 0) continue;
                for (uint32_t b = lane; b < RADIX; b += 32) row[b] = 0;
                __syncwarp();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < ipt) {
                        const uint32_t d = (uint32_t)(k[j] >> (8 * p)) & (RADIX - 1);
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
                constexpr uint32_t PER = RADIX > THREADS ? RADIX / THREADS : 1;
                uint32_t c[PER], sum = 0;
#pragma unroll
                for (uint32_t q = 0; q < PER; ++q) {
                    c[q] = 0;
                    const uint32_t d = tid * PER + q;
                    if (d < RADIX)
                        for (uint32_t w = 0; w < WARPS; ++w) c[q] += s_bin[w * RADIX + d];
                    sum += c[q];
                }
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
                for (uint32_t q = 0; q < PER; ++q) {
                    const uint32_t d = tid * PER + q;
                    if (d < RADIX) {
                        uint32_t r = run;
                        for (uint32_t w = 0; w < WARPS; ++w) {
                            const uint32_t t = s_bin[w * RADIX + d];
                            s_bin[w * RADIX + d] = r;
                            r += t;
                        }
                    }
                    run += c[q];
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < mine) {
                        at[j] += row[(uint32_t)(k[j] >> (8 * p)) & (RADIX - 1)];
                        s_k[at[j]] = k[j];
                        if (PAIRS) s_v[at[j]] = v[j];
                    }
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < mine) {
                        k[j] = s_k[me + j * 32];
                        if (PAIRS) v[j] = s_v[me + j * 32];
                    }
                }
                __syncthreads();
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
