// rs_chunks.cu -- the end of the top-digits order, for items of every width: the
// chunk bounds and the on-chip sorts of the chunks.
#include <algorithm>

#include "rs_bin_sort.cuh"
#include "rs_hist_plan.cuh"
#include "rs_internal.h"

namespace rs {

namespace {

template <typename K, typename V, bool PAIRS, int THREADS, int MIN_BLOCKS>
rs_status launch_chunks(K* keys, V* vals, K* spare_keys, V* spare_vals, const uint32_t* off,
                        const Ctrl* ctrl, uint32_t top_bits, uint32_t key_type, int sm_count,
                        cudaStream_t stream) {
    // (The index of an item takes the place of the bits that its chunk's keys have in
    // common, see TopOrder.)
    using L = BinSortSmem<K, V, PAIRS, THREADS, true>;
    auto kern = k_bin_sort<K, V, PAIRS, THREADS, MIN_BLOCKS, true>;
    static DeviceOnce smem_set;
    const rs_status st = allow_smem_once(kern, L::BYTES, smem_set);
    if (st != RS_OK) return st;
    note_launch_begin(KK_SMALL, stream);
    const cudaError_t e = launch_after_previous(
        kern, dim3(sm_count * MIN_BLOCKS), dim3(THREADS), L::BYTES, stream, keys, vals,
        (const K*)keys, (const V*)vals, off, (const uint32_t*)nullptr, 1,
        (const uint32_t*)&ctrl->chunk_count, ctrl, top_bits, key_type, spare_keys, spare_vals);
    note_launch_end(KK_SMALL, stream);
    return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

template <typename K, typename V, bool PAIRS>
rs_status run(K* keys, V* vals, K* spare_keys, V* spare_vals, uint32_t n, const Ctrl* ctrl,
              uint32_t* off, TopOrder top, uint32_t key_type, cudaStream_t stream) {
    DeviceInfo di;
    const rs_status st = device_info(&di);
    if (st != RS_OK) return st;
    // At most 2^bits chunks by prefix, or one every capacity / 2 items.
    const size_t by_position = sizeof(K) == 8 ? ((size_t)n + top.capacity / 2 - 1) /
                                                    (top.capacity / 2) : 0;
    const size_t most = std::max(size_t(1) << top.bits, by_position);
    const uint32_t ways = top.bits <= 14 ? 32 : 8;
    note_launch_begin(KK_CHUNK_BOUNDS, stream);
    const cudaError_t e = launch_after_previous(
        ways == 32 ? k_chunk_bounds<K, 32> : k_chunk_bounds<K, 8>,
        dim3((uint32_t)((ways * most + 255) / 256)), dim3(256), 0, stream, (const K*)keys,
        (const K*)spare_keys, n, ctrl, top.bits, key_type, off);
    note_launch_end(KK_CHUNK_BOUNDS, stream);
    if (e != cudaSuccess) return RS_ERR_CUDA;
#define RS_CHUNKS(T, B)                                                                     \
    return launch_chunks<K, V, PAIRS, T, B>(keys, vals, spare_keys, spare_vals, off, ctrl,  \
                                            top.bits, key_type, di.sm_count, stream)
    // The shapes that the orders below can ask for: 32-bit items from 2^25 on have larger
    // chunks, wide ones 4608 items at most, and only 64-bit keys come in small arrays.
    constexpr bool WIDE = sizeof(K) == 8 || (PAIRS && sizeof(V) == 8);
    if constexpr (sizeof(K) == 8) {
        if (top.capacity <= 1024) RS_CHUNKS(128, 8);
    }
    if constexpr (WIDE) {
        if (top.capacity <= 2560) RS_CHUNKS(320, 3);
    }
    if (top.capacity <= 4608) RS_CHUNKS(576, 2);
    if constexpr (!WIDE) {
        if (top.capacity <= 8192) RS_CHUNKS(1024, 1);
    }
    return RS_ERR_UNSUPPORTED;  // no shape for it: not reached
#undef RS_CHUNKS
}

}  // namespace

// Chunks of the highest `bits` bits, 2^bits of them, when an average one with seven
// standard deviations on top fits both a CTA of `most` items and an index of `bits`
// bits (a word holds the index in place of those bits).
static TopOrder order_for(size_t n, uint32_t first_bits, uint32_t most) {
    for (uint32_t bits = first_bits; bits <= TOP_MAX_BITS; ++bits) {
        const size_t avg = n >> bits;
        uint32_t root = 1;
        while ((size_t)root * root < avg) ++root;
        const size_t need = avg + 7 * root + 16;
        if (need <= most && need <= (size_t(1) << bits))
            return {bits, need <= 1024 ? 1024u : need <= 2560 ? 2560u : need <= 4608 ? 4608u : 8192u};
    }
    return {0, 0};
}

TopOrder top_order(size_t n) {
    if (n < kTopMinItems) return {0, 0};
    const TopOrder top = order_for(n, 13, 4608);
    return top.bits != 0 ? TopOrder{top.bits, 4608} : order_for(n, TOP_MAX_BITS, 8192);
}

TopOrder top_order_wide(size_t n, bool key64) {
    if (n < (key64 ? kTopMinItems64 : kTopMinItems)) return {0, 0};
    return order_for(n, RADIX_BITS, 4608);
}

rs_status enqueue_chunks(void* keys, void* vals, void* spare_keys, void* spare_vals, uint32_t n,
                         uint32_t key_type, uint32_t val_bytes, const Ctrl* ctrl, uint32_t* off,
                         TopOrder top, cudaStream_t stream) {
    using u32 = uint32_t;
    using u64 = unsigned long long;
#define RS_RUN(K, V, P)                                                                        \
    return run<K, V, P>(static_cast<K*>(keys), static_cast<V*>(vals),                          \
                        static_cast<K*>(spare_keys), static_cast<V*>(spare_vals), n, ctrl, off, \
                        top, key_type, stream)
    if (key_type >= KEY_U64) {
        if (val_bytes == 0) RS_RUN(u64, u32, false);
        if (val_bytes == 4) RS_RUN(u64, u32, true);
        RS_RUN(u64, u64, true);
    }
    if (val_bytes == 0) RS_RUN(u32, u32, false);
    if (val_bytes == 4) RS_RUN(u32, u32, true);
    RS_RUN(u32, u64, true);
#undef RS_RUN
}

}  // namespace rs
