// Row-wise helpers of the tensor-core linears: sums over the splits of k in order, and the gathered rows of routed calls.
#include <cuda_bf16.h>

#include "sm100.cuh"

namespace dmr {

namespace {

// Split-K: Y[row(m)][n] = sum over splits, in split order.
template <bool OUT_F32>
__global__ void __launch_bounds__(256)
splitk_reduce_kernel(const float *__restrict__ partial, int splits, int M, int N, const int32_t *__restrict__ idx,
                     const int32_t *__restrict__ count, void *__restrict__ Y) {
    pdl_wait();  // the partial sums come from the kernel before this one
    pdl_launch_dependents();
    const int rows = count ? min(*count, M) : M;
    if ((N & 3) == 0 && (size_t)rows * (size_t)N < 0x7FFFFFFFull) {
        // four consecutive features per thread: 16-byte loads of every split's sums, one 8- or 16-byte store
        const unsigned nq = (unsigned)N >> 2, total = (unsigned)rows * nq;
        const size_t zstride = (size_t)M * (size_t)N / 4;
        for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
            const unsigned m = i / nq, q = i - m * nq;
            const int row = idx ? idx[m] : (int)m;
            const float4 *p = reinterpret_cast<const float4 *>(partial) + (size_t)m * nq + q;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int z = 0; z < splits; ++z) {  // in split order, as the one-element path below
                const float4 v = p[(size_t)z * zstride];
                s.x += v.x;
                s.y += v.y;
                s.z += v.z;
                s.w += v.w;
            }
            const size_t o = (size_t)row * N + 4u * q;
            if (OUT_F32) {
                *reinterpret_cast<float4 *>(reinterpret_cast<float *>(Y) + o) = s;
            } else {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(s.x, s.y), hi = __floats2bfloat162_rn(s.z, s.w);
                uint2 w;
                w.x = *reinterpret_cast<const uint32_t *>(&lo);
                w.y = *reinterpret_cast<const uint32_t *>(&hi);
                *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(Y) + o) = w;
            }
        }
        return;
    }
    const size_t total = (size_t)rows * N;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(i / N), n = (int)(i % N);
        float s = 0.f;
        for (int z = 0; z < splits; ++z) s += partial[((size_t)z * M + m) * N + n];
        const int row = idx ? idx[m] : m;
        if (OUT_F32) reinterpret_cast<float *>(Y)[(size_t)row * N + n] = s;
        else reinterpret_cast<__nv_bfloat16 *>(Y)[(size_t)row * N + n] = __float2bfloat16_rn(s);
    }
}

// Routed batches: copy the listed rows of X into a dense [Mcap][K] buffer; slots past the count
// are zero-filled so that the tensor core never sees uninitialised memory.
__global__ void __launch_bounds__(256)
gather_rows_kernel(const uint16_t *__restrict__ X, int K, int Mcap, const int32_t *__restrict__ idx,
                   const int32_t *__restrict__ count, int coff, uint16_t *__restrict__ Xg) {
    pdl_wait();  // the row list comes from the kernel before this one
    pdl_launch_dependents();
    const int rows = min(*count - coff, Mcap);
    const int vec_per_row = K / 8;
    const size_t total = (size_t)Mcap * vec_per_row;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int slot = (int)(i / vec_per_row), v = (int)(i % vec_per_row);
        uint4 val = make_uint4(0, 0, 0, 0);
        if (slot < rows) val = *reinterpret_cast<const uint4 *>(X + (size_t)idx[slot] * K + v * 8);
        *reinterpret_cast<uint4 *>(Xg + (size_t)slot * K + v * 8) = val;
    }
}

}  // namespace

dmr_status_t launch_splitk_reduce(const float *partial, int splits, int M, int N, RowSel sel, void *Y, dmr_out_t out,
                                  cudaStream_t st) {
    const size_t total = (size_t)M * N / ((N & 3) == 0 ? 4 : 1);
    int blocks = (int)((total + 255) / 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    if (out == DMR_OUT_F32)
        (void)launch_pdl(splitk_reduce_kernel<true>, dim3((unsigned)blocks), dim3(256), 0, st, partial, splits, M, N, sel.idx, sel.count, Y);
    else
        (void)launch_pdl(splitk_reduce_kernel<false>, dim3((unsigned)blocks), dim3(256), 0, st, partial, splits, M, N, sel.idx, sel.count, Y);
    return check_launch();
}

dmr_status_t launch_gather_rows(const uint16_t *X, int K, int Mcap, const int32_t *idx, const int32_t *count,
                                int coff, uint16_t *Xg, cudaStream_t st) {
    const size_t total = (size_t)Mcap * (K / 8);
    int blocks = (int)((total + 255) / 256);
    if (blocks > 148 * 8) blocks = 148 * 8;
    (void)launch_pdl(gather_rows_kernel, dim3((unsigned)blocks), dim3(256), 0, st, X, K, Mcap, idx, count, coff, Xg);
    return check_launch();
}

}  // namespace dmr
