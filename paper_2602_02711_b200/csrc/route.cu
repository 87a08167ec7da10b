// Route partition: the per-step precision decision r_t (Sec. 3, Eq. 1) arrives as a byte mask,
// 1 = the step needs the high-precision weights (Sec. 4.2, "KL-to-Classification Mapping").
// A stable partition turns it into two ascending row lists, so that each precision's rows can be
// multiplied as one dense batch and written back at their own positions (step order).
#include "sm100.cuh"

namespace dmr {

namespace {

constexpr int kPartThreads = 1024;

// One CTA walks the mask in chunks of 1024 rows; ballots and a 32-entry scan keep the order stable.
__global__ void __launch_bounds__(kPartThreads)
route_partition_kernel(const uint8_t *__restrict__ mask, int M, int32_t *__restrict__ idx_high,
                       int32_t *__restrict__ idx_low, int32_t *__restrict__ counts) {
    __shared__ int warp_high[32];
    __shared__ int base_high_s, base_low_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();  // the lists may still be read, and the mask written, by kernels before this one
    pdl_launch_dependents();
    if (threadIdx.x == 0) {
        base_high_s = 0;
        base_low_s = 0;
    }
    __syncthreads();
    for (int m0 = 0; m0 < M; m0 += kPartThreads) {
        const int m = m0 + threadIdx.x;
        const bool valid = m < M;
        const bool high = valid && mask[m] != 0;
        const unsigned bh = __ballot_sync(0xFFFFFFFFu, high);
        if (lane == 0) warp_high[warp] = __popc(bh);
        __syncthreads();
        int before = 0, total_high = 0;  // high rows in earlier warps of this chunk / in the chunk
        for (int w = 0; w < 32; ++w) {
            const int c = warp_high[w];
            if (w < warp) before += c;
            total_high += c;
        }
        const int chunk_rows = min(kPartThreads, M - m0);
        const int high_rank = before + __popc(bh & ((1u << lane) - 1u));
        const int low_rank = threadIdx.x - high_rank;  // rows before me that are not high
        const int bh0 = base_high_s, bl0 = base_low_s;
        if (valid) {
            if (high) idx_high[bh0 + high_rank] = m;
            else idx_low[bl0 + low_rank] = m;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            base_high_s = bh0 + total_high;
            base_low_s = bl0 + (chunk_rows - total_high);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        counts[0] = base_high_s;
        counts[1] = base_low_s;
    }
}

// Up to 128 rows: every CTA finds the partition by itself (one row per thread) and copies its share of the rows' 16-byte pieces to the two
// halves' buffers; the first one writes the lists.  Latency is all there is to it (the copies are 2 M K bytes: 0.65 MB at M = 64, K = 5120), so
// partition and two gathers are one launch instead of three on two streams.
constexpr int kSplitThreads = 256;
__global__ void __launch_bounds__(kSplitThreads) route_split_kernel(const uint8_t *__restrict__ mask, int M, const uint16_t *__restrict__ X, int K,
                                                                    int32_t *__restrict__ idx_high, int32_t *__restrict__ idx_low,
                                                                    int32_t *__restrict__ counts, uint16_t *__restrict__ Xh, uint16_t *__restrict__ Xl) {
    __shared__ int high_before[5];   // rows of the high half before each warp's 32 rows, and in all
    __shared__ int dest[128];        // slot of a row, high ones as -1 - slot
    pdl_wait();
    pdl_launch_dependents();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool high = t < M && t < 128 && mask[t] != 0;
    const uint32_t votes = __ballot_sync(0xFFFFFFFFu, high);
    if (warp < 4 && lane == 0) high_before[warp + 1] = __popc(votes);
    if (t == 0) high_before[0] = 0;
    __syncthreads();
    if (t == 0)
        for (int i = 1; i < 5; ++i) high_before[i] += high_before[i - 1];
    __syncthreads();
    if (t < M && t < 128) {
        const int h = high_before[warp] + __popc(votes & ((1u << lane) - 1u));
        dest[t] = high ? -1 - h : t - h;
        if (blockIdx.x == 0) {
            if (high) idx_high[h] = t;
            else idx_low[t - h] = t;
        }
    }
    if (blockIdx.x == 0 && t == 0) {
        counts[0] = high_before[4];
        counts[1] = M - high_before[4];
    }
    __syncthreads();
    const int per_row = K / 8;
    for (int i = blockIdx.x * kSplitThreads + t; i < M * per_row; i += gridDim.x * kSplitThreads) {
        const int m = i / per_row, v = i - m * per_row, d = dest[m];
        uint16_t *to = d < 0 ? Xh + (size_t)(-1 - d) * K : Xl + (size_t)d * K;
        reinterpret_cast<uint4 *>(to)[v] = __ldg(reinterpret_cast<const uint4 *>(X + (size_t)m * K) + v);
    }
}

}  // namespace

dmr_status_t launch_route_partition(const uint8_t *mask, int M, int32_t *idx_high, int32_t *idx_low,
                                    int32_t *counts, cudaStream_t st) {
    (void)launch_pdl(route_partition_kernel, dim3(1), dim3(kPartThreads), 0, st, mask, M, idx_high, idx_low, counts);
    return check_launch();
}

dmr_status_t launch_route_split(const uint8_t *mask, int M, const uint16_t *X, int K, int32_t *idx_high, int32_t *idx_low, int32_t *counts,
                                uint16_t *Xh, uint16_t *Xl, cudaStream_t st) {
    int blocks = (M * (K / 8) + kSplitThreads - 1) / kSplitThreads;
    if (blocks > device_sm_count()) blocks = device_sm_count();
    const cudaError_t e = launch_pdl(route_split_kernel, dim3((unsigned)blocks), dim3(kSplitThreads), 0, st, mask, M, X, K, idx_high, idx_low, counts, Xh, Xl);
    if (e != cudaSuccess) return launch_failed(e);
    return check_launch();
}

}  // namespace dmr
