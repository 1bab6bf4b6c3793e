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

// Shared-memory plan of k_bin_sort: the bin words (later the counters of the
// digit passes, later the staged values) and the binned words (later the
// staged keys).
template <typename K, typename V, bool PAIRS, int THREADS, int ITEMS>
struct BinSortSmem {
    static constexpr uint32_t CAP = THREADS * ITEMS;
    static constexpr uint32_t COUNTERS = (THREADS / 32) * RADIX * 4;
    static constexpr uint32_t BINS = CAP * 4 > COUNTERS ? CAP * 4 : COUNTERS;
    static constexpr uint32_t VALS = PAIRS ? CAP * (uint32_t)sizeof(V) : 0;
    static constexpr uint32_t FIRST = BINS > VALS ? BINS : VALS;
    static constexpr size_t BYTES = FIRST + CAP * sizeof(K);
    static_assert(FIRST % 16 == 0, "binned words 16-byte aligned");
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

// ---------------------------------------------------------------------------
// k_bin_sort: sorts arrays of 2 to CAP = THREADS * ITEMS items, one CTA per
// array, each item read from and written to global memory once.  Arrays are
// the segments listed in `list` (every `step`-th entry from it; count in
// *list_count), or with list == nullptr those of the segments 0, 1, ... that
// hold more than single_n items and at most CAP; or with off == nullptr the
// single array [0, single_n).
//
// For an array of m items, nb = 2^bb bins with m <= nb < 2m:
//  1. The keys' bits that differ (an OR over the array) say where the bb
//     highest of them lie; those are the item's bin.  Every item adds one to
//     its bin and keeps the count before it: its place among the bin's items,
//     in no particular order.
//  2. The exclusive prefix over bins gives every bin's first position.  Every
//     item writes the word (key << bb | index) to its bin's next position: the
//     bits shifted out are the same within a bin, or are its bin number, and
//     index < 2^bb.  So the words are distinct, and their order inside a bin is
//     the stable order of the items.
//  3. Every item counts the words of its bin that are smaller than its own:
//     that is its place in the bin, hence its final position.
//  4. Keys and values are staged at their final positions and leave as
//     consecutive stores.
// Step 3 reads sum(c^2) words over the bins' counts c: about 2m for keys that
// spread evenly.  Arrays whose keys crowd into few bins (the sum is known
// after step 2; the line is at BIN_SORT_CROWDED * m) take one stable
// counting pass per 8-bit digit that differs instead: ranks from ballots and
// per-warp counters, items exchanged through shared memory.
//
// What bounds it: shared-memory wavefronts at random bank conflicts, about 27
// per 32 pairs (one counting atomic, one bin read, the word's write, 2 to 3
// reads in step 3 and the staged write, 3.3 each) where four digit passes take
// over 100, and the eight barriers, hidden by the other CTAs on the SM.
// Measured: the 8,900 arrays of 513 to 4096 pairs (15.3 M pairs) among 2^15 short
// ones take 216 us, against 1366 us in four digit passes by 512-thread CTAs; one
// array of 1000 keys takes 6.6 us against 20.4.
// ---------------------------------------------------------------------------
constexpr uint32_t BIN_SORT_CROWDED = 24;

template <typename K, typename V, bool PAIRS, int THREADS, int ITEMS, int MIN_BLOCKS>
__global__ void __launch_bounds__(THREADS, MIN_BLOCKS)
k_bin_sort(K* keys, V* vals, const K* src_keys, const V* src_vals,
           const uint32_t* __restrict__ off, const uint32_t* __restrict__ list, int32_t step,
           const uint32_t* __restrict__ list_count, const Ctrl* __restrict__ ctrl,
           uint32_t single_n, uint32_t key_type) {
    using L = BinSortSmem<K, V, PAIRS, THREADS, ITEMS>;
    constexpr uint32_t WARPS = THREADS / 32;
    static_assert(WARPS <= 32 && L::CAP <= 65535, "one lane per warp total; 16-bit counts");
    pdl_launch_next();
    pdl_wait();  // the kernel before this one (planner, scatter pass) is complete
    extern __shared__ uint4 s_dyn[];
    uint32_t* const s_bin = reinterpret_cast<uint32_t*>(s_dyn);
    V* const s_v = reinterpret_cast<V*>(s_dyn);
    K* const s_w = reinterpret_cast<K*>(reinterpret_cast<char*>(s_dyn) + L::FIRST);
    __shared__ K s_or;
    __shared__ uint32_t s_sum[32], s_sq[32];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    uint32_t count = 1;
    if (off != nullptr) {
        if (ctrl->err != 0) return;
        count = *list_count;
    }
    if (tid == 0) s_or = 0;
    for (uint32_t idx = blockIdx.x; idx < count; idx += gridDim.x) {
        uint32_t lo = 0, m = single_n;
        if (off != nullptr) {
            const uint32_t s = list != nullptr ? list[(ptrdiff_t)idx * step] : idx;
            lo = off[s];
            m = off[s + 1] - lo;
            if (list == nullptr && (m <= single_n || m > L::CAP)) continue;
        }
        // Warp w holds the items [w * 32 * ipt, (w + 1) * 32 * ipt), slot by
        // slot: (warp, slot, lane) order is the input order.
        const uint32_t ipt = (m + THREADS - 1) / THREADS;
        const uint32_t wofs = warp * 32 * ipt + lane;
        const K* const from = src_keys + lo;
        K k[ITEMS];
        K diff = 0;
        const K first = key_to_ordered(from[0], key_type);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            if (j < ipt) {
                const uint32_t i = wofs + j * 32;
                k[j] = i < m ? key_to_ordered(from[i], key_type) : first;
                diff |= k[j] ^ first;
            }
        }
        const uint32_t bb = m > 1 ? 32u - __clz(m - 1) : 1u;
        const uint32_t nb = 1u << bb;
        for (uint32_t b = tid; b < (nb + 3) / 4; b += THREADS)
            reinterpret_cast<uint4*>(s_bin)[b] = make_uint4(0, 0, 0, 0);
        __syncthreads();  // s_or is zero, the bins are free
        diff = warp_or(diff);
        if (lane == 0 && diff != 0) atomicOr(&s_or, diff);
        __syncthreads();
        const K varying = s_or;
        const uint32_t sig = significant_bits(varying);
        const uint32_t shift = sig > bb ? sig - bb : 0u;
        auto bin_of = [&](K x) { return (uint32_t)(x >> shift) & (nb - 1); };

        // ---- 1. count, keeping each item's place among its bin's items ------
        uint32_t at[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            if (j < ipt && wofs + j * 32 < m) at[j] = atomicAdd(&s_bin[bin_of(k[j])], 1u);
        __syncthreads();

        // ---- 2. exclusive prefix over the bins ------------------------------
        // Thread t holds `per` consecutive bins (1, 2, 4, 8 or 16).
        const uint32_t per = nb > THREADS ? nb / THREADS : 1u;
        auto scan_bins = [&](auto per_) {
            constexpr uint32_t PER = decltype(per_)::value;
            const bool mine = tid * PER < nb;
            uint32_t c[PER];
            uint32_t sum = 0, sq = 0;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) c[q] = mine ? s_bin[tid * PER + q] : 0u;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                sum += c[q];
                sq += c[q] * c[q];
            }
            uint32_t x = sum;
#pragma unroll
            for (uint32_t o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            sq = __reduce_add_sync(0xffffffffu, sq);
            if (lane == 31) {
                s_sum[warp] = x;
                s_sq[warp] = sq;
            }
            __syncthreads();
            const uint32_t before = lane < warp ? s_sum[lane] : 0u;
            const uint32_t all = lane < WARPS ? s_sq[lane] : 0u;
            uint32_t run = __reduce_add_sync(0xffffffffu, before) + x - sum;
#pragma unroll
            for (uint32_t q = 0; q < PER; ++q) {
                if (mine) s_bin[tid * PER + q] = run | (c[q] << 16);  // first position, count
                run += c[q];
            }
            return __reduce_add_sync(0xffffffffu, all);
        };
        uint32_t sq;
        if (per == 1) sq = scan_bins(std::integral_constant<uint32_t, 1>{});
        else if (per == 2) sq = scan_bins(std::integral_constant<uint32_t, 2>{});
        else if (per == 4 || ITEMS == 4) sq = scan_bins(std::integral_constant<uint32_t, 4>{});
        else if (per == 8 || ITEMS == 8) sq = scan_bins(std::integral_constant<uint32_t, 8>{});
        else sq = scan_bins(std::integral_constant<uint32_t, ITEMS>{});
        if (tid == 0) s_or = 0;  // for the next array
        __syncthreads();

        V v[PAIRS ? ITEMS : 1];
        if (sq <= BIN_SORT_CROWDED * m) {
            // ---- 2. the words, bin by bin ---------------------------------
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t i = wofs + j * 32;
                if (j < ipt && i < m) {
                    const uint32_t e = s_bin[bin_of(k[j])];
                    s_w[(e & 0xffffu) + at[j]] = (k[j] << bb) | (K)i;
                    at[j] = e;
                }
            }
            if (PAIRS) {
#pragma unroll
                for (int j = 0; j < ITEMS; ++j)
                    if (j < ipt && wofs + j * 32 < m) v[j] = src_vals[lo + wofs + j * 32];
            }
            __syncthreads();
            // ---- 3. every item's place in its bin -------------------------
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t i = wofs + j * 32;
                if (j < ipt && i < m) {
                    const uint32_t c = at[j] >> 16;
                    uint32_t pos = at[j] & 0xffffu;
                    if (c > 1) {
                        const K w = (k[j] << bb) | (K)i;
                        const K* const bin = s_w + pos;
                        for (uint32_t q = 0; q < c; ++q) pos += bin[q] < w ? 1u : 0u;
                    }
                    at[j] = pos;
                }
            }
            __syncthreads();
            // ---- 4. staged in order, stored in order -----------------------
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                if (j < ipt && wofs + j * 32 < m) {
                    s_w[at[j]] = k[j];
                    if (PAIRS) s_v[at[j]] = v[j];
                }
            }
            __syncthreads();
            for (uint32_t i = tid; i < m; i += THREADS) {
                keys[lo + i] = key_from_ordered(s_w[i], key_type);
                if (PAIRS) vals[lo + i] = s_v[i];
            }
            __syncthreads();  // shared memory is free for the next array
        } else {
            // ---- digit passes ------------------------------------------------
            // Items stay in registers; a pass moves them to their new slots
            // through shared memory (keys through s_w, then values over the
            // counters, which are free by then).
            const uint32_t lt = lanemask_lt();
            uint32_t* const row = s_bin + warp * RADIX;
            if (PAIRS) {
#pragma unroll
                for (int j = 0; j < ITEMS; ++j)
                    if (j < ipt && wofs + j * 32 < m) v[j] = src_vals[lo + wofs + j * 32];
            }
            for (uint32_t p = 0; p < sizeof(K); ++p) {
                if (((varying >> (8 * p)) & (RADIX - 1)) == 0) continue;
                for (uint32_t b = lane; b < RADIX; b += 32) row[b] = 0;
                __syncwarp();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < ipt) {
                        const uint32_t d = (uint32_t)(k[j] >> (8 * p)) & (RADIX - 1);
                        const uint32_t live = prefix_lanes(wofs - lane + j * 32, m);
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
                    if (j < ipt && wofs + j * 32 < m) {
                        at[j] += row[(uint32_t)(k[j] >> (8 * p)) & (RADIX - 1)];
                        s_w[at[j]] = k[j];
                    }
                }
                __syncthreads();
#pragma unroll
                for (int j = 0; j < ITEMS; ++j) {
                    if (j < ipt && wofs + j * 32 < m) {
                        k[j] = s_w[wofs + j * 32];
                        if (PAIRS) s_v[at[j]] = v[j];
                    }
                }
                __syncthreads();
                if (PAIRS) {
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j)
                        if (j < ipt && wofs + j * 32 < m) v[j] = s_v[wofs + j * 32];
                    __syncthreads();
                }
            }
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) {
                const uint32_t i = wofs + j * 32;
                if (j < ipt && i < m) {
                    keys[lo + i] = key_from_ordered(k[j], key_type);
                    if (PAIRS) vals[lo + i] = v[j];
                }
            }
        }
    }
}

}  // namespace rs
