// rs_segmented_wide.cuh -- the per-segment digit histograms of 64-bit keys, for the
// segmented sort of wide items (64-bit keys, or 32-bit keys carrying 64-bit values).
// The large segments take the scatter passes (k_onesweep<..., SEG>) with the
// items' widths, as the 32-bit segmented sort does; the others the bin sort.
#pragma once

#include "rs_device.cuh"

namespace rs {

// ---------------------------------------------------------------------------
// k_seg_hist64: the eight digit histograms of every large segment of 64-bit
// keys, added into hist[ordinal][8][256] (zeroed by the caller).  One CTA
// per SM takes a contiguous run of tiles (consecutive tiles mostly share a
// segment), counts into a CTA-private shared histogram with shared atomics,
// and adds it to the segment's global histogram when the segment changes.
// Also clears the first scatter pass's status array.  TYPED: keys are mapped
// onto their ordered words first.
// ---------------------------------------------------------------------------
constexpr uint32_t SEG_HIST64_THREADS = 1024;

template <bool TYPED>
__global__ void __launch_bounds__(SEG_HIST64_THREADS, 1)
k_seg_hist64(const unsigned long long* __restrict__ keys, const Ctrl* __restrict__ ctrl,
             const uint4* __restrict__ tile_geo, uint32_t* __restrict__ hist,
             uint4* __restrict__ clear, uint32_t clear_vec4, uint32_t key_type) {
    __shared__ uint32_t s_h[PASSES64 * RADIX];
    constexpr uint32_t T = SEG_HIST64_THREADS;
    const uint32_t tid = threadIdx.x;
    for (uint32_t i = blockIdx.x * T + tid; i < clear_vec4; i += gridDim.x * T)
        clear[i] = make_uint4(0, 0, 0, 0);
    if (ctrl->err != 0) return;
    const uint32_t tiles = ctrl->seg_tiles;
    const uint32_t per = (tiles + gridDim.x - 1) / gridDim.x;
    const uint32_t t_lo = blockIdx.x * per;
    const uint32_t t_hi = t_lo + per < tiles ? t_lo + per : tiles;
    if (t_lo >= t_hi) return;
    for (uint32_t i = tid; i < PASSES64 * RADIX; i += T) s_h[i] = 0;
    __syncthreads();
    auto flush = [&](uint32_t seg) {
        __syncthreads();
        for (uint32_t bin = tid; bin < PASSES64 * RADIX; bin += T) {
            const uint32_t c = s_h[bin];
            if (c) atomicAdd(hist + (size_t)seg * PASSES64 * RADIX + bin, c);
            s_h[bin] = 0;
        }
        __syncthreads();
    };
    uint32_t cur = 0xffffffffu;
    for (uint32_t t = t_lo; t < t_hi; ++t) {
        const uint4 g = tile_geo[t];  // the same for every thread of the CTA
        if (g.w != cur) {
            if (cur != 0xffffffffu) flush(cur);
            cur = g.w;
        }
        for (uint32_t i = tid; i < g.y; i += T) {
            unsigned long long k = __ldcs(keys + g.x + i);
            if (TYPED) k = key_to_ordered(k, key_type);
#pragma unroll
            for (uint32_t p = 0; p < PASSES64; ++p)
                atomicAdd(&s_h[p * RADIX + ((uint32_t)(k >> (8u * p)) & (RADIX - 1))], 1u);
        }
    }
    flush(cur);
}

}  // namespace rs
