// rs_internal.h -- host-side interface between the C ABI (rs_api.cu) and the
// kernel launchers (rs_sort.cu, rs_onesweep_*.cu).  Not installed, not part
// of the ABI.
#pragma once

#include <atomic>
#include <utility>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/rs.h"

namespace rs {

struct Ctrl;

// Kernel kinds, for launch counting and per-kind event timing.
enum KernelKind : int {
    KK_HIST = 0,
    KK_PLAN = 1,
    KK_ONESWEEP = 2,
    KK_SMALL = 3,
    KK_SEG_PLAN = 4,
    KK_SEG_HIST = 5,
    KK_SEG_SCAN = 6,
    KK_SEG_ONESWEEP = 7,
    KK_WARP = 8,
    KK_D11_UP = 9,
    KK_D11_SCAN = 10,
    KK_D11_DOWN = 11,
    KK_CHUNK_BOUNDS = 12,
    KK_CLEAR = 13,
    KK_COUNT
};
const char* kernel_kind_name(int kind);

// Called around every kernel launch by the launchers.
void note_launch_begin(int kind, cudaStream_t stream);
void note_launch_end(int kind, cudaStream_t stream);

// Tile shapes of the scatter kernel that this build instantiates:
// X(index, threads, items per thread, CTAs per SM the register budget is
// sized for, look-back window in status words).  The launchers and the host
// tables are both generated from this one list.
#define RS_TILE_SHAPES(X)   \
    X(0, 512, 16, 1, 32)    \
    X(1, 512, 8, 2, 16)     \
    X(2, 256, 16, 2, 32)    \
    X(3, 384, 13, 2, 6)     \
    X(4, 384, 12, 2, 8)     \
    X(5, 1024, 8, 1, 32)    \
    X(6, 384, 18, 2, 8)

struct TileConfig {
    int threads;
    int items;
    int min_blocks;  // CTAs per SM the register budget is sized for
    int window;      // look-back window (status words read per round trip)
};
#define RS_COUNT_SHAPE(I, T, J, B, W) +1
constexpr int NUM_TILE_CONFIGS = 0 RS_TILE_SHAPES(RS_COUNT_SHAPE);
#undef RS_COUNT_SHAPE
extern const TileConfig kTileConfigs[NUM_TILE_CONFIGS];
int smallest_tile();
// Sorts of typed keys run their scatter passes with this shape (the default
// of large arrays); only it is compiled with the key maps.
constexpr int kTypedShape = 3;

// Per size class tuning (chosen by the autotuner): tile shapes (indices into
// kTileConfigs), the largest array / segment sorted on chip (small_max; up to warp_max
// in the smallest CTAs), and the on-chip sorts taken (small_bits: 8, the bin sort, or
// 4, the counting sorts by 4-bit digits).
struct ClassKnobs {
    int tile_pairs;
    int tile_keys;
    int tile_seg;
    int small_max;
    int warp_max;
    int small_bits;
    int msd;        // 1: whole arrays may take the MSD-first or the top-digits order
    int digits;     // 8: four 8-bit passes; 11: three 11/11/10-bit passes (rs_digits11.cu)
                    // for unsigned keys, when the caller's workspace holds their buffers
};
// The MSD-first order sorts the buckets of the highest digit on chip: by a CTA of
// 5120 items for arrays of up to 256 * 4600 items, of 8192 up to 256 * 7400 items
// (the largest bucket of evenly spread keys stays seven or more standard deviations below).
constexpr uint32_t kMsdShortItems = 256u * 4600u;
constexpr uint32_t kMsdMaxItems = 256u * 7400u;
// Large arrays may take the top-digits order: two scatter passes, then chunks of the
// keys' `bits` highest bits sorted on chip by a CTA of `capacity` items (rs_chunks.cu).
// bits = 0: not tried.  32-bit keys from kTopMinItems on (tried below, it took 382 us
// instead of 389 for 2^24 pairs, but 574 instead of 538 for 24 million), 64-bit keys, which
// save six passes of eight, from kTopMinItems64.  Above 495,976,448 items (271,187,968 wide
// ones) the chunks of 16 bits no longer fit a CTA.
constexpr uint32_t kTopMinItems = 1u << 25;
constexpr uint32_t kTopMinItems64 = 1u << 14;
struct TopOrder {
    uint32_t bits, capacity;
};
TopOrder top_order(size_t n);
TopOrder top_order_wide(size_t n, bool key64);
// The end of that order, once the passes are enqueued: off is a table of 2^bits + 1 words
// in the workspace; the spare arrays are the other buffers of the passes.
rs_status enqueue_chunks(void* keys, void* vals, void* spare_keys, void* spare_vals, uint32_t n,
                         uint32_t key_type, uint32_t val_bytes, const Ctrl* ctrl, uint32_t* off,
                         TopOrder top, cudaStream_t stream);
// Size classes by item count (whole array; for a segmented sort the average
// segment): <= 2^13, <= 2^16, <= 2^20, <= 2^24, <= 2^28, larger.
constexpr int NUM_SIZE_CLASSES = 6;
int size_class(size_t items);

// Host-side knobs shared by every launch.
struct Knobs {
    ClassKnobs cls[NUM_SIZE_CLASSES];
    uint32_t spin_limit;     // polls per look-back wait before ERR_TIMEOUT
    uint32_t debug;          // DBG_* bits
    int hist_ctas_per_sm;
    int hist_mode;           // HIST_ATOMIC / HIST_LEADER / HIST_MATCH
    // Typed keys: sorts of at least this many items launch two instances of
    // every scatter pass (the passes that need no key map run without it);
    // smaller ones launch only the mapping instance, which runs every pass.
    uint32_t typed_split_min;
    int d11_shape;           // tile shape of the 11-bit-digit sort's scatter kernel
    int pdl;                 // 1: the plan and scatter kernels launch as programmatic dependents
};
Knobs& knobs();
// Whether a typed sort of n items launches two instances of every scatter
// pass (see Knobs::typed_split_min).
inline bool typed_split(size_t n) { return n >= knobs().typed_split_min; }

// Host-side checks shared by the sort entry points: size, null pointers,
// 4-byte alignment, keys and values not overlapping.
rs_status check_sort_args(const uint32_t* keys, const uint32_t* vals, size_t n);

// Per-device facts cached on first use.
struct DeviceInfo {
    int sm_count;
    uint32_t* sticky;        // device address of the sticky error word
};
rs_status device_info(DeviceInfo* out);

// Workspace layout of an unsegmented sort of n items.
struct Layout {
    size_t ctrl, status0, status1, alt_keys, alt_vals, msd_off, total;
    uint32_t tiles;          // tiles of the smallest tile shape (status sizing)
    bool wide_status;        // 64-bit status words (n >= 2^30)
};
Layout layout_for(size_t n, bool pairs);
// Workspace of the whole-array sorts of n items: the 8-bit layout, or the
// 11-bit one's when n's size class takes that order and it is larger.
size_t sort_workspace_bytes(size_t n, bool pairs);

// Enqueue the whole sort of n items (1 <= n < 2^32) on `stream`, using the
// caller's workspace (at least layout_for(n, pairs).total bytes).
rs_status enqueue_sort(uint32_t* keys, uint32_t* vals, uint32_t n, cudaStream_t stream,
                       void* workspace, size_t workspace_bytes, uint32_t key_type = 0);

// Alg. 2's local MSD pass: one stable counting-sort pass of n (1 <= n <
// 2^32) keys (with values when vals != nullptr) by digit 3 from the inputs
// into the outputs, and the 257 bucket offsets; workspace as for a sort.
rs_status enqueue_msd_partition(const uint32_t* keys, const uint32_t* vals, uint32_t n,
                                uint32_t* out_keys, uint32_t* out_vals, uint32_t* bucket_off,
                                cudaStream_t stream, void* workspace, size_t workspace_bytes);

// The sort with 11-bit digits (three passes of 11, 11 and 10 bits;
// rs_digits11.cu): two alternate key (and value) buffers, per-chunk digit
// counts of at most kD11MaxChunks chunks, and the 2048 bucket totals.
constexpr uint32_t kD11MaxChunks = 1024;
struct Layout11 {
    size_t alt_keys[2], alt_vals[2], counts, totals, total;
    uint32_t max_chunks;
};
Layout11 layout11(size_t n, bool pairs);
int d11_shape_count();
rs_status enqueue_sort11(uint32_t* keys, uint32_t* vals, uint32_t n, cudaStream_t stream,
                         void* workspace, size_t workspace_bytes);

// Wide items: 64-bit keys (eight passes; key_type KEY_U64, KEY_I64 or
// KEY_F64) carrying no, 32-bit or 64-bit values (val_bytes 0, 4 or 8), and
// 32-bit keys (KEY_U32, KEY_I32, KEY_F32) carrying 64-bit values.  Arrays of up to
// kWideSmallMax items are sorted on chip, longer ones take scatter passes.
Layout layout_wide(size_t n, bool key64, uint32_t val_bytes);
rs_status enqueue_sort_wide(void* keys, void* vals, uint32_t n, uint32_t key_type,
                            uint32_t val_bytes, cudaStream_t stream, void* workspace,
                            size_t workspace_bytes);
// Scatter-pass tiles of the wide sorts: 384 threads, items per thread.
constexpr int kWideThreads = 384;
constexpr int kWideItems64 = 7;     // 64-bit keys, no or 32-bit values
constexpr int kWideItems64V64 = 6;  // 64-bit keys, 64-bit values
constexpr int kWideItems32V64 = 7;  // 32-bit keys, 64-bit values
// One scatter pass of 64-bit keys (rs_sort64.cu); wide = 64-bit status words.
rs_status launch_pass_k64(uint32_t key_type, uint32_t val_bytes, bool wide,
                          unsigned long long* ka, void* va, unsigned long long* kb, void* vb,
                          uint32_t n, uint32_t pass, Ctrl* ctrl, uint32_t* sticky, void* status,
                          void* status_clear, cudaStream_t stream);

// Enqueue the digit histograms of n keys into hist[4 * 256] (zeroed first).
rs_status enqueue_histograms(const uint32_t* keys, uint32_t n, uint32_t* hist,
                             cudaStream_t stream);
// The same, added into hist (zeroed by the caller), counting the digits of
// the ordered words of typed keys, and clearing clear_bytes at `clear`.
// (after_clear: enqueue_clear was the last launch on the stream.)
rs_status enqueue_hist4(const uint32_t* keys, uint32_t n, uint32_t* hist, void* clear,
                        size_t clear_bytes, uint32_t key_type, cudaStream_t stream,
                        bool after_clear = false);
// Zeroes the control block, and more_bytes (a multiple of 16) at `more`.
rs_status enqueue_clear(Ctrl* ctrl, cudaStream_t stream, void* more = nullptr,
                        size_t more_bytes = 0);
// The plan kernel (rs_hist_plan.cuh), for keys of NPASS digits.
struct PlanArgs;
template <int NPASS> rs_status enqueue_plan(const PlanArgs& plan, cudaStream_t stream);

// Segmented scatter passes: per-tile geometry and per-segment bucket bases
// built on the device, and an upper bound of the tile count for the launch.
struct SegView {
    const uint4* tile_geo = nullptr;
    const uint32_t* gofs = nullptr;
    uint32_t max_tiles = 0;
    bool routed = false;  // tiles placed by each segment's order (k_seg_scan)
};

// Scatter-pass launchers, one per value flavour (separate translation units);
// seg == nullptr for the unsegmented sort.
// key_type: KEY_U32, KEY_I32 or KEY_F32 (rs_device.cuh).
// slot: the plan entry of the launch (the pass, or MSD_SLOT).
rs_status launch_onesweep_keys(int cfg, bool wide, uint32_t* ka, uint32_t* kb, uint32_t n,
                               uint32_t pass, uint32_t slot, Ctrl* ctrl, uint32_t* sticky,
                               void* status, void* status_clear, const SegView* seg,
                               uint32_t key_type, cudaStream_t stream);
rs_status launch_onesweep_pairs(int cfg, bool wide, uint32_t* ka, uint32_t* va, uint32_t* kb,
                                uint32_t* vb, uint32_t n, uint32_t pass, uint32_t slot,
                                Ctrl* ctrl, uint32_t* sticky, void* status, void* status_clear,
                                const SegView* seg, uint32_t key_type, cudaStream_t stream);

// One-CTA sorts on chip of the segments 0 .. *count - 1 (count on the device) of at
// most bucket_capacity(long_buckets) items each, read from src_keys / src_vals.
// bits: 8, the bin sort (rs_bin_sort.cuh); 4, eight counting passes of 4-bit digits.
uint32_t bucket_capacity(bool long_buckets);
rs_status launch_bucket_sorts(uint32_t* keys, uint32_t* vals, const uint32_t* src_keys,
                              const uint32_t* src_vals, const uint32_t* off,
                              const uint32_t* count, const Ctrl* ctrl, bool long_buckets,
                              int bits, uint32_t key_type, cudaStream_t stream);
// The bin sort of wide items (rs_small_wide.cu): of the single array [0, n), n <=
// kWideSmallMax, and of the segments of up to as many items that are listed by size.
constexpr uint32_t kWideSmallMax = 4096;
rs_status launch_single_wide(void* keys, void* vals, uint32_t n, uint32_t key_type,
                             uint32_t val_bytes, cudaStream_t stream);
rs_status launch_lists_wide(void* keys, void* vals, const uint32_t* off, const uint32_t* tiny_list,
                            const uint32_t* small_list, uint32_t entries, const Ctrl* ctrl,
                            uint32_t key_type, uint32_t val_bytes, cudaStream_t stream);
// One-CTA sorts on chip of *count ranges (first item, items) at `runs`, of at most 4096
// items each.
rs_status launch_run_sorts(uint32_t* keys, uint32_t* vals, const uint32_t* src_keys,
                           const uint32_t* src_vals, const uint32_t* runs, const uint32_t* count,
                           const Ctrl* ctrl, int bits, uint32_t key_type, cudaStream_t stream);
// The segments listed by size (rs_bin_sort.cuh list_small) in tiny_list and
// small_list of `entries` entries each, in place: one launch per size up to
// max_items.
rs_status launch_small_lists(uint32_t* keys, uint32_t* vals, const uint32_t* off,
                             const uint32_t* tiny_list, const uint32_t* small_list,
                             uint32_t entries, const Ctrl* ctrl, uint32_t max_items, int bits,
                             uint32_t key_type, cudaStream_t stream);
// The same sort of the single array [0, n), n <= small_sort_capacity().
rs_status launch_single_sort(uint32_t* keys, uint32_t* vals, uint32_t n, int bits,
                             uint32_t key_type, cudaStream_t stream);
uint32_t small_sort_capacity();

// The same sorts of the tiny segments listed by the planner (at most
// warp_sort_capacity() items each): by a CTA of two warps, or with bits = 4 one warp.
rs_status launch_tiny_list(uint32_t* keys, uint32_t* vals, const uint32_t* off,
                           const uint32_t* tiny_list, const Ctrl* ctrl, int bits,
                           uint32_t key_type, cudaStream_t stream);
uint32_t warp_sort_capacity();

// Workspace layout of a segmented sort of n items in num_segments segments.
struct SegLayout {
    size_t ctrl, status0, status1, alt_keys, alt_vals, tile_geo, tiny_list, small_list, large_first,
        gofs, total;
    // The 32-bit sorts' parts for segments that take the MSD-first order; a
    // workspace of `total` bytes, without them, has all take the LSD passes.
    size_t route_geo, runs, routed_total;
    uint32_t max_tiles, max_large;
};
SegLayout seg_layout_for(size_t n, bool pairs, uint32_t num_segments);
// Segmented sorts of wide items (64-bit keys, or 32-bit keys with 64-bit
// values; rs_segmented_wide.cu).
SegLayout seg_layout_wide(size_t n, bool key64, uint32_t val_bytes, uint32_t num_segments);
rs_status enqueue_sort_segmented_wide(void* keys, void* vals, uint32_t n,
                                      const uint32_t* offsets, uint32_t num_segments,
                                      uint32_t key_type, uint32_t val_bytes, cudaStream_t stream,
                                      void* workspace, size_t workspace_bytes);
rs_status enqueue_sort_segmented(uint32_t* keys, uint32_t* vals, uint32_t n,
                                 const uint32_t* offsets, uint32_t num_segments,
                                 cudaStream_t stream, void* workspace, size_t workspace_bytes,
                                 uint32_t key_type = 0);

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Launch `kern` on `stream`; with knobs().pdl set, as a programmatic
// dependent of the kernel before it on the stream, so that it becomes
// resident while that kernel finishes (the kernel calls pdl_wait() before
// reading that kernel's output).
template <typename... Params, typename... Args>
cudaError_t launch_after_previous(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = knobs().pdl ? 1u : 0u;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// A first kernel: beside the clearing of its counts (it waits for that before it uses
// them), when that is the launch before.
template <typename... Params, typename... Args>
cudaError_t launch_hist(bool after_clear, void (*kern)(Params...), dim3 grid, dim3 block,
                        size_t smem, cudaStream_t stream, Args&&... args) {
    if (after_clear)
        return launch_after_previous(kern, grid, block, smem, stream, std::forward<Args>(args)...);
    kern<<<grid, block, smem, stream>>>(std::forward<Args>(args)...);
    return cudaPeekAtLastError();
}

// One bit per device (ordinal < 64) for one-time host setup of a kernel
// (its shared-memory limit), safe when several host threads enqueue sorts.
struct DeviceOnce {
    std::atomic<uint64_t> bits{0};
    bool done(int dev) const { return (bits.load(std::memory_order_acquire) >> dev) & 1u; }
    void mark(int dev) { bits.fetch_or(uint64_t(1) << dev, std::memory_order_release); }
};

// Raise the dynamic shared-memory limit of `kern` to `bytes` once per device.
template <typename Kern>
rs_status allow_smem_once(Kern kern, size_t bytes, DeviceOnce& once) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return RS_ERR_CUDA;
    if (!once.done(dev)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
            cudaSuccess)
            return RS_ERR_CUDA;
        once.mark(dev);
    }
    return RS_OK;
}

}  // namespace rs
