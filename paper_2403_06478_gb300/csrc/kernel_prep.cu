// Batch preparation on the device: validate every pair, route it to the warp
// kernel or (band too wide) to the block kernel, and order the warp kernel's
// work queue longest-first.
//
// Ordering follows the paper's performance model (Section 4.5): the work of a
// pair is about Cells = Antidiags x Band_width, and the slowest warps dominate
// (the MAX over warps in Table 1).  Uneven bucketing (Section 4.4) spreads the
// longest tasks over different warps; here the persistent kernel's queue hands
// out pairs in decreasing predicted work (longest-processing-time first), so
// the long pairs start first and the short ones fill the tail.  The sort is a
// counting sort over 256 quarter-octave buckets of predicted cells.
#include "agatha_dev.cuh"

namespace agatha {

constexpr int PREP_THREADS = 256;
constexpr int N_BUCKETS = 256;
constexpr int PREP_SMALL_THREADS = 1024;

// Bucket 0 holds the largest predicted work.
__device__ __forceinline__ int32_t work_bucket(int32_t tlen, int32_t qlen, int32_t w) {
    const uint64_t est = predicted_cells(tlen, qlen, w);
    const int32_t lg = 63 - __clzll(est);                    // floor(log2)
    const int32_t frac = lg >= 2 ? (int32_t)((est >> (lg - 2)) & 3) : 0;
    int32_t key = lg * 4 + frac;                              // 4 buckets per octave
    key = key > N_BUCKETS - 1 ? N_BUCKETS - 1 : key;
    return N_BUCKETS - 1 - key;
}

__global__ void prep_classify_kernel(const DevBatch *__restrict__ d_batch, int32_t sort) {
    const DevBatch B = *d_batch;
    if (threadIdx.x == 0) mark_step_begin(B.counters);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < B.n_pairs;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!pair_valid(B, i)) {
            atomicExch(&B.counters[CTR_ERR], DEV_ERR_BAD_PAIR);
            write_empty_result(B.out + i);
            continue;
        }
        const int32_t tl = B.t_len[i], ql = B.q_len[i];
        const int32_t w = effective_w(B.params.w, tl, ql);
        if (w > B.warp_w_max || (B.narrow_w_max > 0 && w <= B.narrow_w_max)) {
            // too wide for the warp kernel (the block kernel's list), or a band
            // the narrower frame takes (its own list; never both in one batch)
            const int32_t k = atomicAdd(&B.counters[CTR_NWIDE], 1);
            B.wide_order[k] = (int32_t)i;
            continue;
        }
        if (sort) atomicAdd((unsigned long long *)&B.bucket_hist[work_bucket(tl, ql, w)], 1ull);
        else atomicAdd(&B.counters[CTR_NWARP], 1);
    }
}

// Exclusive scan of the bucket histogram (one block); bucket_hist[b] becomes
// the first queue position of bucket b.
__global__ void prep_scan_kernel(const DevBatch *__restrict__ d_batch) {
    const DevBatch B = *d_batch;
    __shared__ int64_t s[N_BUCKETS];
    const int t = threadIdx.x;
    s[t] = B.bucket_hist[t];
    __syncthreads();
    for (int o = 1; o < N_BUCKETS; o <<= 1) {
        const int64_t v = t >= o ? s[t - o] : 0;
        __syncthreads();
        s[t] += v;
        __syncthreads();
    }
    const int64_t incl = s[t];
    B.bucket_hist[t] = incl - B.bucket_hist[t];
    if (t == N_BUCKETS - 1) B.counters[CTR_NWARP] = (int32_t)incl;
}

__global__ void prep_scatter_kernel(const DevBatch *__restrict__ d_batch) {
    const DevBatch B = *d_batch;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < B.n_pairs;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!pair_valid(B, i)) continue;
        const int32_t tl = B.t_len[i], ql = B.q_len[i];
        const int32_t w = effective_w(B.params.w, tl, ql);
        if (w > B.warp_w_max || (B.narrow_w_max > 0 && w <= B.narrow_w_max)) continue;
        const int32_t b = work_bucket(tl, ql, w);
        const int64_t pos = (int64_t)atomicAdd((unsigned long long *)&B.bucket_hist[b], 1ull);
        B.order[pos] = (int32_t)i;
    }
}

// All of it, and the clearing of the counters and the histogram, for a small
// batch in one block: the launches were longer than their work.
__global__ void __launch_bounds__(PREP_SMALL_THREADS) prep_small_kernel(const DevBatch *__restrict__ d_batch,
                                                                        int32_t sort) {
    __shared__ int32_t hist[N_BUCKETS], n_wide, n_warp, err;
    const DevBatch B = *d_batch;
    const int t = threadIdx.x;
    if (t < N_BUCKETS) hist[t] = 0;
    if (t == 0) n_wide = n_warp = 0, err = DEV_ERR_NONE;
    if (t < CTR_COUNT) B.counters[t] = 0;
    __syncthreads();
    if (t == 0) mark_step_begin(B.counters);
    const auto bucket = [&](int64_t i, int32_t &w) {
        const int32_t tl = B.t_len[i], ql = B.q_len[i];
        w = effective_w(B.params.w, tl, ql);
        return work_bucket(tl, ql, w);
    };
    const auto listed = [&](int32_t w) {                      // as prep_classify_kernel
        return w > B.warp_w_max || (B.narrow_w_max > 0 && w <= B.narrow_w_max);
    };
    for (int64_t i = t; i < B.n_pairs; i += PREP_SMALL_THREADS) {
        if (!pair_valid(B, i)) {
            err = DEV_ERR_BAD_PAIR;
            write_empty_result(B.out + i);
            continue;
        }
        int32_t w;
        const int32_t b = bucket(i, w);
        if (listed(w)) B.wide_order[atomicAdd(&n_wide, 1)] = (int32_t)i;
        else if (sort) atomicAdd(&hist[b], 1);
        else atomicAdd(&n_warp, 1);
    }
    __syncthreads();
    if (t == 0) {
        B.counters[CTR_NWIDE] = n_wide;
        B.counters[CTR_ERR] = err;
        if (!sort) B.counters[CTR_NWARP] = n_warp;
    }
    if (!sort) return;
    if (t < 32) {                                             // exclusive scan, 8 buckets a lane
        int32_t v[N_BUCKETS / 32], sum = 0;
        for (int i = 0; i < N_BUCKETS / 32; ++i) sum += v[i] = hist[t * (N_BUCKETS / 32) + i];
        int32_t at = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t x = __shfl_up_sync(0xffffffffu, at, o);
            if (t >= o) at += x;
        }
        if (t == 31) B.counters[CTR_NWARP] = at;
        at -= sum;
        for (int i = 0; i < N_BUCKETS / 32; ++i) {
            hist[t * (N_BUCKETS / 32) + i] = at;
            at += v[i];
        }
    }
    __syncthreads();
    for (int64_t i = t; i < B.n_pairs; i += PREP_SMALL_THREADS) {
        if (!pair_valid(B, i)) continue;
        int32_t w;
        const int32_t b = bucket(i, w);
        if (!listed(w)) B.order[atomicAdd(&hist[b], 1)] = (int32_t)i;
    }
    __syncthreads();
    if (t < N_BUCKETS) B.bucket_hist[t] = hist[t];
}

// Clears the counters (and the histogram, unless hist is null), then validates,
// routes and (sort) orders the pairs.  One launch up to PREP_SMALL pairs,
// where one SM is no slower than two memsets and three launches (256 pairs:
// 3.6 us instead of 12; 4,096: 9 of 16).
cudaError_t launch_prep(const DevBatch *d_batch, int64_t n_pairs, int32_t sort, int32_t *counters, int64_t *hist,
                        cudaStream_t s, int n_sm) {
    if (prep_small(n_pairs) && hist) {
        prep_small_kernel<<<1, PREP_SMALL_THREADS, 0, s>>>(d_batch, sort);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(counters, 0, CTR_COUNT * sizeof(int32_t), s);
    if (e == cudaSuccess && hist) e = cudaMemsetAsync(hist, 0, N_BUCKETS * sizeof(int64_t), s);
    if (e != cudaSuccess) return e;
    // a fixed grid (grid-stride loops) so one captured graph serves any batch size
    const int64_t blocks = (int64_t)(n_sm > 0 ? n_sm : 1) * 4;
    prep_classify_kernel<<<(unsigned)blocks, PREP_THREADS, 0, s>>>(d_batch, sort);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess || !sort) return err;
    prep_scan_kernel<<<1, N_BUCKETS, 0, s>>>(d_batch);
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    prep_scatter_kernel<<<(unsigned)blocks, PREP_THREADS, 0, s>>>(d_batch);
    return cudaGetLastError();
}

}  // namespace agatha
