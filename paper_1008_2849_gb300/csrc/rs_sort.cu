// rs_sort.cu -- histogram and plan kernels, workspace layout and the
// enqueue sequence of one unsegmented sort.
#include <algorithm>

#include "rs_internal.h"
#include "rs_hist_plan.cuh"

namespace rs {

// Must list the shapes of RS_TILE_SHAPES (rs_onesweep_launch.cuh) in order.
#define RS_SHAPE_ENTRY(I, T, J, B, W) {T, J, B, W},
const TileConfig kTileConfigs[NUM_TILE_CONFIGS] = {RS_TILE_SHAPES(RS_SHAPE_ENTRY)};
#undef RS_SHAPE_ENTRY

int smallest_tile() {
    int t = kTileConfigs[0].threads * kTileConfigs[0].items;
    for (int i = 1; i < NUM_TILE_CONFIGS; ++i)
        if (kTileConfigs[i].threads * kTileConfigs[i].items < t)
            t = kTileConfigs[i].threads * kTileConfigs[i].items;
    return t;
}

constexpr int HIST_THREADS = 512;

Layout layout_for(size_t n, bool pairs) {
    Layout L{};
    const size_t tile = (size_t)smallest_tile();
    L.tiles = (uint32_t)((n + tile - 1) / tile);
    L.wide_status = n >= (size_t(1) << 30);
    const size_t status_bytes = (size_t)L.tiles * RADIX * (L.wide_status ? 8 : 4);
    size_t off = 0;
    L.ctrl = off;
    off = align_up(off + sizeof(Ctrl), 256);
    L.status0 = off;
    off = align_up(off + status_bytes, 256);
    L.status1 = off;
    off = align_up(off + status_bytes, 256);
    L.alt_keys = off;
    off = align_up(off + n * sizeof(uint32_t), 256);
    L.alt_vals = off;
    if (pairs) off = align_up(off + n * sizeof(uint32_t), 256);
    L.msd_off = off;  // MSD-first order: bucket offsets
    off = align_up(off + (RADIX + 1) * sizeof(uint32_t), 256);
    L.total = off;
    return L;
}

rs_status enqueue_clear(Ctrl* ctrl, cudaStream_t stream, void* more, size_t more_bytes) {
    const size_t vecs = more_bytes / sizeof(uint4);
    const uint32_t grid = (uint32_t)std::min<size_t>(1 + vecs / 8192, 512);
    note_launch_begin(KK_CLEAR, stream);
    k_clear_ctrl<<<grid, 1024, 0, stream>>>(reinterpret_cast<uint4*>(ctrl),
                                            static_cast<uint4*>(more), vecs);
    note_launch_end(KK_CLEAR, stream);
    return cudaPeekAtLastError() == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

rs_status enqueue_hist4(const uint32_t* keys, uint32_t n, uint32_t* hist, void* clear,
                        size_t clear_bytes, uint32_t key_type, cudaStream_t stream,
                        bool after_clear) {
    DeviceInfo di;
    rs_status st = device_info(&di);
    if (st != RS_OK) return st;
    const uint32_t vec4 = (uint32_t)(n / 4);
    uint32_t blocks = (uint32_t)(di.sm_count * knobs().hist_ctas_per_sm);
    const uint32_t needed = (vec4 + 63) / 64 / (HIST_THREADS / 32) + 1;  // 64 vectors per warp
    if (blocks > needed) blocks = needed;
    if (blocks < 1) blocks = 1;
    if (knobs().hist_mode == HIST_COLUMNS) {
        // Eight columns (two CTAs per SM, two 16-byte loads a thread) up to 2^21
        // keys, then 32: 2^20 uniform keys sort in 37.1 us instead of 38.9, 2^18 in
        // 31.4 instead of 32.1; from 2^22 on the 32-column reads are faster.
        const bool few = n <= (1u << 21), typed = key_type != KEY_U32;
        constexpr int T8 = 512, T32 = 1024;
        const size_t smem = (few ? HIST_COL_WORDS<8> : HIST_COL_WORDS<32>) * sizeof(uint32_t);
        auto kern = few ? (typed ? k_hist4_cols<T8, 8, true> : k_hist4_cols<T8, 8, false>)
                        : (typed ? k_hist4_cols<T32, 32, true> : k_hist4_cols<T32, 32, false>);
        static DeviceOnce smem_set[4];  // per instance
        st = allow_smem_once(kern, smem, smem_set[(few ? 2 : 0) + (typed ? 1 : 0)]);
        if (st != RS_OK) return st;
        uint32_t grid = (uint32_t)di.sm_count * (few ? 2u : 1u);
        const uint32_t need = few ? (vec4 + 2 * T8 - 1) / (2 * T8) : (vec4 + T32 - 1) / T32;
        if (grid > need) grid = need > 0 ? need : 1;
        note_launch_begin(KK_HIST, stream);
        const cudaError_t e = launch_hist(
            after_clear, kern, dim3(grid), dim3(few ? T8 : T32), smem, stream, keys, n, hist,
            static_cast<uint4*>(clear), (uint32_t)(clear_bytes / sizeof(uint4)), key_type);
        note_launch_end(KK_HIST, stream);
        return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
    }
    const bool typed = key_type != KEY_U32;
    auto kern = typed ? k_hist4<HIST_THREADS, HIST_LEADER, true>
                      : k_hist4<HIST_THREADS, HIST_LEADER, false>;
    switch (knobs().hist_mode) {
    case HIST_ATOMIC:
        kern = typed ? k_hist4<HIST_THREADS, HIST_ATOMIC, true>
                     : k_hist4<HIST_THREADS, HIST_ATOMIC, false>;
        break;
    case HIST_MATCH:
        kern = typed ? k_hist4<HIST_THREADS, HIST_MATCH, true>
                     : k_hist4<HIST_THREADS, HIST_MATCH, false>;
        break;
    default: break;
    }
    note_launch_begin(KK_HIST, stream);
    kern<<<blocks, HIST_THREADS, 0, stream>>>(keys, n, hist, static_cast<uint4*>(clear),
                                              (uint32_t)(clear_bytes / sizeof(uint4)), key_type);
    note_launch_end(KK_HIST, stream);
    return cudaPeekAtLastError() == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}

template <int NPASS>
rs_status enqueue_plan(const PlanArgs& plan, cudaStream_t stream) {
    const bool top = plan.top_bits != 0;
    auto kern = top ? k_plan<NPASS, true> : k_plan<NPASS, false>;
    size_t smem = 0;
    if (top) {
        static DeviceOnce smem_set;
        const rs_status st = allow_smem_once(kern, TOP_PLAN_SMEM, smem_set);
        if (st != RS_OK) return st;
        smem = top_plan_smem(plan.n, plan.top_bits, NPASS == PASSES64);
    }
    note_launch_begin(KK_PLAN, stream);
    const cudaError_t e = launch_after_previous(kern, dim3(1), dim3(1024), smem, stream, plan);
    note_launch_end(KK_PLAN, stream);
    return e == cudaSuccess ? RS_OK : RS_ERR_CUDA;
}
template rs_status enqueue_plan<PASSES>(const PlanArgs&, cudaStream_t);
template rs_status enqueue_plan<PASSES64>(const PlanArgs&, cudaStream_t);

rs_status enqueue_histograms(const uint32_t* keys, uint32_t n, uint32_t* hist,
                             cudaStream_t stream) {
    if (cudaMemsetAsync(hist, 0, PASSES * RADIX * sizeof(uint32_t), stream) != cudaSuccess)
        return RS_ERR_CUDA;
    return enqueue_hist4(keys, n, hist, nullptr, 0, KEY_U32, stream);
}

rs_status enqueue_msd_partition(const uint32_t* keys, const uint32_t* vals, uint32_t n,
                                uint32_t* out_keys, uint32_t* out_vals, uint32_t* bucket_off,
                                cudaStream_t stream, void* workspace, size_t workspace_bytes) {
    const bool pairs = vals != nullptr;
    const Layout L = layout_for(n, pairs);
    if (workspace == nullptr || workspace_bytes < L.total || ((uintptr_t)workspace & 255u))
        return RS_ERR_INVALID_ARG;
    DeviceInfo di;
    rs_status st = device_info(&di);
    if (st != RS_OK) return st;
    char* ws = static_cast<char*>(workspace);
    Ctrl* ctrl = reinterpret_cast<Ctrl*>(ws + L.ctrl);
    void* status = ws + L.status0;
    const size_t status_bytes = L.status1 - L.status0;
    if (cudaMemsetAsync(ctrl, 0, sizeof(Ctrl), stream) != cudaSuccess) return RS_ERR_CUDA;
    st = enqueue_hist4(keys, n, &ctrl->hist[0][0], status, status_bytes, KEY_U32, stream);
    if (st != RS_OK) return st;
    note_launch_begin(KK_PLAN, stream);
    k_msd_plan<<<1, RADIX, 0, stream>>>(ctrl, n, bucket_off);
    note_launch_end(KK_PLAN, stream);
    if (cudaPeekAtLastError() != cudaSuccess) return RS_ERR_CUDA;
    const ClassKnobs& ck = knobs().cls[size_class(n)];
    // The scatter kernels read the source through the plan's direction
    // (A -> B) and never write it.
    uint32_t* src_k = const_cast<uint32_t*>(keys);
    uint32_t* src_v = const_cast<uint32_t*>(vals);
    return pairs ? launch_onesweep_pairs(ck.tile_pairs, L.wide_status, src_k, src_v, out_keys,
                                         out_vals, n, PASSES - 1, MSD_SLOT, ctrl, di.sticky,
                                         status, nullptr, nullptr, KEY_U32, stream)
                 : launch_onesweep_keys(ck.tile_keys, L.wide_status, src_k, out_keys, n,
                                        PASSES - 1, MSD_SLOT, ctrl, di.sticky, status, nullptr,
                                        nullptr, KEY_U32, stream);
}

rs_status enqueue_sort(uint32_t* keys, uint32_t* vals, uint32_t n, cudaStream_t stream,
                       void* workspace, size_t workspace_bytes, uint32_t key_type) {
    if (key_type > KEY_F32) return RS_ERR_INVALID_ARG;
    const bool pairs = vals != nullptr;
    const Layout L = layout_for(n, pairs);
    if (workspace == nullptr || workspace_bytes < L.total || ((uintptr_t)workspace & 255u))
        return RS_ERR_INVALID_ARG;
    DeviceInfo di;
    rs_status st = device_info(&di);
    if (st != RS_OK) return st;
    const ClassKnobs& ck = knobs().cls[size_class(n)];
    // A single small array takes one CTA.
    if (n <= (uint32_t)ck.small_max && n <= small_sort_capacity())
        return launch_single_sort(keys, vals, n, ck.small_bits, key_type, stream);
    // Three passes of 11/11/10-bit digits, where the size class takes them
    // and the caller's workspace holds their buffers.
    if (ck.digits == 11 && key_type == KEY_U32 && workspace_bytes >= layout11(n, pairs).total)
        return enqueue_sort11(keys, vals, n, stream, workspace, workspace_bytes);
    char* ws = static_cast<char*>(workspace);
    Ctrl* ctrl = reinterpret_cast<Ctrl*>(ws + L.ctrl);
    void* status[2] = {ws + L.status0, ws + L.status1};
    const size_t status_bytes = L.status1 - L.status0;
    uint32_t* alt_k = reinterpret_cast<uint32_t*>(ws + L.alt_keys);
    uint32_t* alt_v = pairs ? reinterpret_cast<uint32_t*>(ws + L.alt_vals) : nullptr;

    // MSD-first order (Alg. 2): tried for arrays that can split into 256
    // buckets the one-CTA sort takes; the plan decides on the device from the
    // digit-3 histogram, so the launch sequence stays fixed.  Large arrays: the
    // top-digits order likewise.
    const bool msd = ck.msd != 0 && n <= kMsdMaxItems;
    const bool long_buckets = n > kMsdShortItems;
    const TopOrder top = ck.msd != 0 ? top_order(n) : TopOrder{0, 0};
    uint32_t* msd_off = reinterpret_cast<uint32_t*>(ws + L.msd_off);
    const PlanArgs plan{ctrl, keys, n, key_type, bucket_capacity(long_buckets),
                        msd ? msd_off : nullptr, top.bits, 0u, top.capacity};

    st = enqueue_clear(ctrl, stream);
    if (st != RS_OK) return st;
    st = enqueue_hist4(keys, n, &ctrl->hist[0][0], status[0], status_bytes, key_type, stream, true);
    if (st != RS_OK) return st;
    st = enqueue_plan<PASSES>(plan, stream);
    if (st != RS_OK) return st;

    const int cfg = pairs ? ck.tile_pairs : ck.tile_keys;
    for (uint32_t p = 0; p < PASSES; ++p) {
        void* cur = status[p & 1];
        void* next = p + 1 < PASSES ? status[(p + 1) & 1] : nullptr;
        // Pass 3 is the MSD-first order's only pass (into the alternate
        // buffers) when the plan chose it.
        const uint32_t kt = key_type | (msd && p == PASSES - 1 ? ROLE_MSD_TOO : 0u);
        st = pairs ? launch_onesweep_pairs(cfg, L.wide_status, keys, vals, alt_k, alt_v, n, p, p,
                                           ctrl, di.sticky, cur, next, nullptr, kt, stream)
                   : launch_onesweep_keys(cfg, L.wide_status, keys, alt_k, n, p, p, ctrl, di.sticky,
                                          cur, next, nullptr, kt, stream);
        if (st != RS_OK) return st;
    }
    if (msd)  // every bucket on chip, back into the caller's arrays
        return launch_bucket_sorts(keys, vals, alt_k, alt_v, msd_off, &ctrl->small_count, ctrl,
                                   long_buckets, ck.small_bits, key_type, stream);
    // The array is sorted by its top 16 bits (or finished, if the plan chose the
    // four passes); the status words are free for the table of chunks.
    if (top.bits != 0)
        return enqueue_chunks(keys, vals, alt_k, alt_v, n, key_type, pairs ? 4u : 0u, ctrl,
                              static_cast<uint32_t*>(status[0]), top, stream);
    return RS_OK;
}

}  // namespace rs
