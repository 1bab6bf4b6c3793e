// rs_small.cu -- host launchers of the on-chip sorts of 32-bit keys with no or 32-bit
// values: the bin sort (rs_bin_sort.cuh), or the 4-bit counting passes of rs_small.cuh.
#include "rs_bin_sort.cuh"
#include "rs_internal.h"
#include "rs_small.cuh"

namespace rs {

namespace {

// What a one-CTA sort works on: arrays listed on the device, or a single one.
struct SmallWork {
    uint32_t *keys, *vals;
    const uint32_t *src_keys, *src_vals, *off, *list;
    int32_t step;
    const uint32_t* list_count;
    const Ctrl* ctrl;
    uint32_t single_n;  // off == nullptr: the array's items
    uint32_t key_type;
};

// A single array takes one CTA, a list as many as fit the GPU `per_sm` to an SM.
rs_status grid_of(const SmallWork& w, uint32_t per_sm, uint32_t* grid) {
    DeviceInfo di;
    const rs_status st = device_info(&di);
    if (st == RS_OK) *grid = w.off == nullptr ? 1u : (uint32_t)di.sm_count * per_sm;
    return st;
}

template <bool PAIRS, int THREADS, int MIN_BLOCKS>
rs_status launch_bin_shape(const SmallWork& w, cudaStream_t stream) {
    using L = BinSortSmem<uint32_t, uint32_t, PAIRS, THREADS, false>;
    auto kern = k_bin_sort<uint32_t, uint32_t, PAIRS, THREADS, MIN_BLOCKS>;
    static DeviceOnce smem_set;
    rs_status st = allow_smem_once(kern, L::BYTES, smem_set);
    if (st != RS_OK) return st;
    uint32_t grid = 0;
    st = grid_of(w, MIN_BLOCKS, &grid);
    if (st != RS_OK) return st;
    note_launch_begin(KK_SMALL, stream);
    const cudaError_t e = launch_after_previous(
        kern, dim3(grid), dim3(THREADS), L::BYTES, stream, w.keys, w.vals, w.src_keys, w.src_vals,
        w.off, w.list, w.step, w.list_count, w.ctrl, w.single_n, w.key_type,
        (uint32_t*)nullptr, (uint32_t*)nullptr);
    note_launch_end(KK_SMALL, stream);
    return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

template <int THREADS, int ITEMS, bool PAIRS>
rs_status launch_small_shape4(const SmallWork& w, cudaStream_t stream) {
    constexpr uint32_t CAP = THREADS * ITEMS;
    constexpr size_t SMEM = ((PAIRS ? 4u : 2u) * CAP + (THREADS / 32) * 16u) * sizeof(uint32_t);
    auto kern = k_small_sort<THREADS, ITEMS, 4, PAIRS>;
    static DeviceOnce smem_set;
    rs_status st = allow_smem_once(kern, SMEM, smem_set);
    if (st != RS_OK) return st;
    uint32_t grid = 0;
    st = grid_of(w, 4, &grid);
    if (st != RS_OK) return st;
    note_launch_begin(KK_SMALL, stream);
    const cudaError_t e = launch_after_previous(kern, dim3(grid), dim3(THREADS), SMEM, stream,
                                                w.keys, w.vals, w.src_keys, w.src_vals, w.off,
                                                w.list, w.step, w.list_count, w.ctrl, w.single_n,
                                                w.key_type);
    note_launch_end(KK_SMALL, stream);
    return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

// The CTA for arrays of at most max_items items: 128 threads up to 1024, 512 up
// to 4096, 1024 up to 8192 (eight items a thread).  A single array of up to 1024
// takes 512 threads: fewer items a thread, a shorter chain.
template <bool PAIRS>
rs_status launch_small_size(uint32_t max_items, int bits, const SmallWork& w,
                            cudaStream_t stream) {
    if (bits == 4)
        return max_items <= SMALL_MID_MAX ? launch_small_shape4<256, 16, PAIRS>(w, stream)
                                          : launch_small_shape4<512, 16, PAIRS>(w, stream);
    if (max_items <= SMALL_SHORT_MAX && w.off != nullptr)
        return launch_bin_shape<PAIRS, 128, 8>(w, stream);
    if (max_items <= SMALL_MID_MAX) return launch_bin_shape<PAIRS, 512, 2>(w, stream);
    return launch_bin_shape<PAIRS, 1024, 1>(w, stream);
}

rs_status launch_small_any(uint32_t max_items, int bits, const SmallWork& w,
                           cudaStream_t stream) {
    return w.vals != nullptr ? launch_small_size<true>(max_items, bits, w, stream)
                             : launch_small_size<false>(max_items, bits, w, stream);
}

template <bool PAIRS>
rs_status launch_warp4(const SmallWork& w, cudaStream_t stream) {
    using L = WarpSortSmem<WARP_SORT_ITEMS, 4, PAIRS>;
    auto kern = k_warp_sort<WARP_SORT_ITEMS, 4, PAIRS>;
    static DeviceOnce smem_set;
    rs_status st = allow_smem_once(kern, L::BYTES, smem_set);
    if (st != RS_OK) return st;
    uint32_t grid = 0;
    st = grid_of(w, 3, &grid);
    if (st != RS_OK) return st;
    note_launch_begin(KK_WARP, stream);
    const cudaError_t e = launch_after_previous(kern, dim3(grid), dim3(WARP_SORT_THREADS), L::BYTES,
                                                stream, w.keys, w.vals, w.off, w.list, w.ctrl,
                                                w.key_type);
    note_launch_end(KK_WARP, stream);
    return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

}  // namespace

uint32_t small_sort_capacity() { return 8192; }
uint32_t warp_sort_capacity() { return 32 * WARP_SORT_ITEMS; }

uint32_t bucket_capacity(bool long_buckets) { return long_buckets ? 8192 : 5120; }

rs_status launch_bucket_sorts(uint32_t* keys, uint32_t* vals, const uint32_t* src_keys,
                              const uint32_t* src_vals, const uint32_t* off,
                              const uint32_t* count, const Ctrl* ctrl, bool long_buckets,
                              int bits, uint32_t key_type, cudaStream_t stream) {
    const SmallWork w{keys, vals, src_keys, src_vals, off, nullptr, 1, count, ctrl, 0, key_type};
    if (long_buckets || bits == 4) return launch_small_any(small_sort_capacity(), bits, w, stream);
    return vals != nullptr ? launch_bin_shape<true, 640, 2>(w, stream)
                           : launch_bin_shape<false, 640, 2>(w, stream);
}

rs_status launch_run_sorts(uint32_t* keys, uint32_t* vals, const uint32_t* src_keys,
                           const uint32_t* src_vals, const uint32_t* runs, const uint32_t* count,
                           const Ctrl* ctrl, int bits, uint32_t key_type, cudaStream_t stream) {
    const SmallWork w{keys, vals, src_keys, src_vals, runs, runs, 0, count, ctrl, 0, key_type};
    return launch_small_any(SMALL_MID_MAX, bits, w, stream);
}

rs_status launch_small_lists(uint32_t* keys, uint32_t* vals, const uint32_t* off,
                             const uint32_t* tiny_list, const uint32_t* small_list,
                             uint32_t entries, const Ctrl* ctrl, uint32_t max_items, int bits,
                             uint32_t key_type, cudaStream_t stream) {
    const struct {
        const uint32_t* list;
        int step;
        const uint32_t* count;
        uint32_t below, max;
    } sizes[] = {
        {small_list, 1, &ctrl->small_count, 0, SMALL_SHORT_MAX},
        {small_list + entries - 1, -1, &ctrl->mid_count, SMALL_SHORT_MAX, SMALL_MID_MAX},
        {tiny_list + entries - 1, -1, &ctrl->big_count, SMALL_MID_MAX, small_sort_capacity()},
    };
    for (const auto& c : sizes) {
        if (max_items <= c.below) break;
        const SmallWork w{keys, vals, keys, vals, off, c.list, c.step, c.count, ctrl, 0,
                          key_type};
        const rs_status st = launch_small_any(c.max, bits, w, stream);
        if (st != RS_OK) return st;
    }
    return RS_OK;
}

rs_status launch_single_sort(uint32_t* keys, uint32_t* vals, uint32_t n, int bits,
                             uint32_t key_type, cudaStream_t stream) {
    if (n > small_sort_capacity()) return RS_ERR_INVALID_ARG;
    const SmallWork w{keys, vals, keys, vals, nullptr, nullptr, 1, nullptr, nullptr, n, key_type};
    return launch_small_any(n, bits, w, stream);
}

rs_status launch_tiny_list(uint32_t* keys, uint32_t* vals, const uint32_t* off,
                           const uint32_t* tiny_list, const Ctrl* ctrl, int bits,
                           uint32_t key_type, cudaStream_t stream) {
    const SmallWork w{keys, vals, keys, vals, off, tiny_list, 1, &ctrl->tiny_count, ctrl, 0,
                      key_type};
    if (bits == 4)
        return vals != nullptr ? launch_warp4<true>(w, stream) : launch_warp4<false>(w, stream);
    return vals != nullptr ? launch_bin_shape<true, 64, 16>(w, stream)
                           : launch_bin_shape<false, 64, 16>(w, stream);
}

}  // namespace rs
