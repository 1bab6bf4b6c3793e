// rs_small_wide.cu -- host launchers of the bin sort (rs_bin_sort.cuh) for small
// arrays and segments of wide items: 64-bit keys, or 32-bit keys with 64-bit values.
//
// Segments up to 512, 1024 and 4096 items take CTAs of 64, 128 and 512 threads, as
// many on an SM as their shared memory admits; 8192 64-bit keys with 64-bit values
// do not fit a CTA, and longer segments take the scatter passes.  Against one warp
// for up to 256 items and eight scatter passes for the rest, 2^15 segments of 2 to
// 4096 items (17.6 M 64-bit keys with 32-bit values) take 0.40 ms a call, 2.12 before;
// 2^14 of 64 to 512 items, 0.12 and 0.83.  4096 of 256 to 65536, of which most items
// keep the passes: 2.88 and 3.15.
#include "rs_bin_sort.cuh"
#include "rs_internal.h"

namespace rs {

namespace {

template <typename K, typename V, bool PAIRS, int THREADS, int MIN_BLOCKS>
rs_status launch(K* keys, V* vals, const uint32_t* off, const uint32_t* list, int step,
                 const uint32_t* count, const Ctrl* ctrl, uint32_t single_n, uint32_t key_type,
                 cudaStream_t stream) {
    using L = BinSortSmem<K, V, PAIRS, THREADS, false>;
    static_assert(L::BYTES + 2048 <= 232448, "shared memory plan exceeds one CTA's limit");
    auto kern = k_bin_sort<K, V, PAIRS, THREADS, MIN_BLOCKS>;
    static DeviceOnce smem_set;
    rs_status st = allow_smem_once(kern, L::BYTES, smem_set);
    if (st != RS_OK) return st;
    DeviceInfo di;
    st = device_info(&di);
    if (st != RS_OK) return st;
    const uint32_t grid = off == nullptr ? 1u : (uint32_t)(di.sm_count * MIN_BLOCKS);
    note_launch_begin(KK_SMALL, stream);
    const cudaError_t e = launch_after_previous(
        kern, dim3(grid), dim3(THREADS), L::BYTES, stream, keys, vals, (const K*)keys,
        (const V*)vals, off, list, (int32_t)step, count, ctrl, single_n, key_type, (K*)nullptr,
        (V*)nullptr);
    note_launch_end(KK_SMALL, stream);
    return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

template <typename K, typename V, bool PAIRS>
rs_status lists(K* keys, V* vals, const uint32_t* off, const uint32_t* tiny_list,
                const uint32_t* small_list, uint32_t entries, const Ctrl* ctrl, uint32_t key_type,
                cudaStream_t stream) {
    rs_status st = launch<K, V, PAIRS, 64, 12>(keys, vals, off, tiny_list, 1, &ctrl->tiny_count,
                                               ctrl, 0, key_type, stream);
    if (st != RS_OK) return st;
    st = launch<K, V, PAIRS, 128, 7>(keys, vals, off, small_list, 1, &ctrl->small_count, ctrl, 0,
                                     key_type, stream);
    if (st != RS_OK) return st;
    return launch<K, V, PAIRS, 512, 2>(keys, vals, off, small_list + entries - 1, -1,
                                       &ctrl->mid_count, ctrl, 0, key_type, stream);
}

}  // namespace

#define RS_WIDE(F, ...)                                                                          \
    do {                                                                                         \
        using u32 = uint32_t;                                                                    \
        using u64 = unsigned long long;                                                          \
        if (key_type < KEY_U64)                                                                  \
            return F<u32, u64, true>(static_cast<u32*>(keys), static_cast<u64*>(vals),           \
                                     __VA_ARGS__);                                               \
        if (val_bytes == 0)                                                                      \
            return F<u64, u32, false>(static_cast<u64*>(keys), (u32*)nullptr, __VA_ARGS__);      \
        if (val_bytes == 4)                                                                      \
            return F<u64, u32, true>(static_cast<u64*>(keys), static_cast<u32*>(vals),           \
                                     __VA_ARGS__);                                               \
        return F<u64, u64, true>(static_cast<u64*>(keys), static_cast<u64*>(vals), __VA_ARGS__); \
    } while (0)

template <typename K, typename V, bool PAIRS>
static rs_status single(K* keys, V* vals, uint32_t n, uint32_t key_type, cudaStream_t stream) {
    return launch<K, V, PAIRS, 512, 2>(keys, vals, nullptr, nullptr, 1, nullptr, nullptr, n,
                                       key_type, stream);
}

rs_status launch_single_wide(void* keys, void* vals, uint32_t n, uint32_t key_type,
                             uint32_t val_bytes, cudaStream_t stream) {
    if (n > SMALL_MID_MAX) return RS_ERR_INVALID_ARG;
    RS_WIDE(single, n, key_type, stream);
}

rs_status launch_lists_wide(void* keys, void* vals, const uint32_t* off, const uint32_t* tiny_list,
                            const uint32_t* small_list, uint32_t entries, const Ctrl* ctrl,
                            uint32_t key_type, uint32_t val_bytes, cudaStream_t stream) {
    RS_WIDE(lists, off, tiny_list, small_list, entries, ctrl, key_type, stream);
}

}  // namespace rs
