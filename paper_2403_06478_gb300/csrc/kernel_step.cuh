// Score kernels with a maximum and a termination test on every anti-diagonal,
// for scorings whose Z-drop threshold leaves the lazy blocks no room
// (lazy_pays in agatha_dev.cuh).  There lazy_drive would run its masked step,
// which keeps one copy of the code for both parities and every edge, nearly
// everywhere: 250 ALU instructions per 16-slot anti-diagonal against the 114 of
// the bulk step here.  One GB300, whole calls, lazy blocks against this
// kernel at a threshold of 30 with minimap2's ONT scoring: 8,000 pairs of 600 bp
// at w = 100 4.21 and 1.37 ms, 1,500 ONT-like pairs of 5 kbp at w = 500 17.2 and
// 6.2, int32 lanes 27.5 and 15.1; the assembly preset (b = 19, threshold 200)
// at w = 500, 5,000 pairs of 2 kbp, 10.7 and 7.4.  One warp per pair; blocks of
// four warps take pairs from one queue, longest first (no tiers: with three to
// six blocks on an SM the chip is full).
#pragma once

#include "kernel_warp16.cuh"

namespace agatha {

// int32 lanes.
template <int C>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS)
warp_step_kernel(const DevBatch *__restrict__ d_batch, int32_t use_fast, int32_t list) {
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31;
    const WorkList L = work_list(B, list);
    if (list == WARP_LIST_OVERFLOW && L.end == 0) return;        // nearly always
    bool had = blockIdx.x == 0;
    for (;;) {
        int32_t k = 0;
        if (lane == 0) k = L.begin + atomicAdd(L.head, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= L.end) break;
        had = true;
        const int32_t pair = L.items ? L.items[k] : k;
        if (!L.items && (!pair_valid(B, pair) || !warp_takes(B, pair))) continue;
        WarpPair<C> wp;
        wp.run(B, pair, lane, use_fast != 0);
    }
    if (lane == 0 && had) mark_step_end(B.counters);
}

template <int C>
cudaError_t launch_step_c(const DevBatch *d_batch, int n_blocks, cudaStream_t s, int use_fast, int list) {
    warp_step_kernel<C><<<n_blocks, WARP_BLOCK_THREADS, 0, s>>>(d_batch, use_fast, list);
    return cudaGetLastError();
}

template <int C>
int occupancy_step_c() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, warp_step_kernel<C>, WARP_BLOCK_THREADS, 0) != cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

// 16-bit lanes, cut for MINB resident blocks per SM.
template <int C, int MINB>
__global__ void __launch_bounds__(WARP_BLOCK_THREADS, MINB)
warp16_step_kernel(const DevBatch *__restrict__ d_batch, int32_t use_fast, int32_t list) {
    // the larger register budget of each slot count also runs the head on the
    // bulk step and defers the edge steps' arg-max
    constexpr bool HIGH = C == 4 ? MINB == 4 : (C >= 20 ? MINB == 2 : MINB == 3);
    __shared__ Cold16 cold[WARP_BLOCK_THREADS / 32];
    const DevBatch B = *d_batch;
    const int lane = threadIdx.x & 31;
    const WorkList L = work_list(B, list);
    bool had = blockIdx.x == 0;
    for (;;) {
        int32_t k = 0;
        if (lane == 0) k = L.begin + atomicAdd(L.head, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= L.end) break;
        had = true;
        const int32_t pair = L.items ? L.items[k] : k;
        if (!L.items && (!pair_valid(B, pair) || !warp_takes(B, pair))) continue;
        WarpPair16<C, (MINB < 4 && C <= 16) || MINB < 3, true, false, true, 1, HIGH, HIGH> wp(cold[threadIdx.x >> 5]);
        if (!wp.run(B, pair, lane, use_fast != 0) && lane == 0) {
            const int32_t slot = atomicAdd(&B.counters[CTR_NOVF], 1);
            B.ovf_list[slot] = pair;
        }
    }
    if (lane == 0 && had) mark_step_end(B.counters);
}

// priority: of the launch on its stream (see launch_warp16_prio).
template <int C, int MINB>
cudaError_t launch_step16_c(const DevBatch *d_batch, int n_blocks, cudaStream_t s, int use_fast, int list,
                            const int *priority) {
    if (!priority) {
        warp16_step_kernel<C, MINB><<<n_blocks, WARP_BLOCK_THREADS, 0, s>>>(d_batch, use_fast, list);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_blocks);
    cfg.blockDim = dim3(WARP_BLOCK_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributePriority;
    attr[0].val.priority = *priority;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, warp16_step_kernel<C, MINB>, d_batch, use_fast, list);
}

template <int C, int MINB>
int occupancy_step16_c() {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, warp16_step_kernel<C, MINB>, WARP_BLOCK_THREADS, 0) !=
        cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

}  // namespace agatha
