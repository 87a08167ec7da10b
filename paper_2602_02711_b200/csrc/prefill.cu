// Low-bit linears of prefill size: the activations are prepared here, the product is pair.cu's.  Prefill is a dense contraction (its
// cost is folded into the per-token latency, App. "Latency coefficients"), so it belongs on the tensor cores.
//
// Operand precision.  The MMA runs in fp16 x fp16 -> fp32 (kind::f16) instead of bf16: a bf16 A
// operand would round every dequantized weight to 8 significant bits (1.5e-3 rms relative error of
// the outputs, uncomfortably close to the 2e-3 acceptance bound), fp16 keeps 11 (1.8e-4).  To stay
// inside fp16's range whatever the inputs, a preparation kernel rescales every activation row by a
// power of two (row maximum into [2^13, 2^14): exact for all elements within 2^-27 of the maximum)
// and the unpack threads rescale a feature's scales by the power of two of its largest one; the
// epilogue multiplies the two powers of two back in (exact).
#include <cuda_bf16.h>

#include "sm100.cuh"

namespace dmr {

namespace {

// Activation preparation: Xh[slot][k] = fp16(X[row(slot)][k] * 2^-e), xscale[slot] = 2^e, with e chosen
// per row so that the row's largest magnitude lands in [2^13, 2^14).  Slots past the valid count
// (routed calls) are zero-filled.  `idx` / `count`: the rows to take and how many (nullptr = all).
__device__ __forceinline__ uint32_t row_max_bits(const uint4 &q, uint32_t mx) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a0 = w[i] & 0x7FFFu, a1 = (w[i] >> 16) & 0x7FFFu;
        if (a0 < 0x7F80u) mx = max(mx, a0);  // largest FINITE magnitude (bf16 patterns order like magnitudes)
        if (a1 < 0x7F80u) mx = max(mx, a1);
    }
    return mx;
}

__device__ __forceinline__ uint4 to_f16_scaled(const uint4 &q, float down, float down2) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float f0 = __uint_as_float(w[i] << 16) * down * down2;
        const float f1 = __uint_as_float(w[i] & 0xFFFF0000u) * down * down2;
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(o[i]) : "f"(f1), "f"(f0));
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// One CTA of 256 threads per slot (grid-stride over slots); CH = 16-byte chunks a thread keeps in
// registers between the two passes (CH * 256 * 8 >= K), so the row is read from memory once.
template <int CH>
__global__ void __launch_bounds__(256)
xprep_kernel(const uint16_t *__restrict__ X, int K, int Mcap, const int32_t *__restrict__ idx,
             const int32_t *__restrict__ count, uint16_t *__restrict__ Xh, float *__restrict__ xscale) {
    __shared__ uint32_t warp_max[8];
    pdl_wait();               // nothing of the stream's earlier work is read or overwritten before this
    pdl_launch_dependents();  // the GEMM behind this kernel may set itself up meanwhile
    const int rows = count ? min(*count, Mcap) : Mcap;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nv = K / 8;
    for (int slot = blockIdx.x; slot < Mcap; slot += gridDim.x) {
        uint4 *dst = reinterpret_cast<uint4 *>(Xh + (size_t)slot * K);
        if (slot >= rows) {
            for (int v = threadIdx.x; v < nv; v += 256) dst[v] = make_uint4(0, 0, 0, 0);
            if (threadIdx.x == 0) xscale[slot] = 1.f;
            continue;
        }
        const uint4 *src = reinterpret_cast<const uint4 *>(X + (size_t)(idx ? idx[slot] : slot) * K);
        uint4 keep[CH];
        uint32_t mx = 0;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int v = c * 256 + threadIdx.x;
            keep[c] = v < nv ? __ldg(src + v) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int c = 0; c < CH; ++c) mx = row_max_bits(keep[c], mx);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
        __syncthreads();  // warp_max of the previous slot has been read by everyone
        if (lane == 0) warp_max[warp] = mx;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w) mx = max(mx, warp_max[w]);
        int eb = (int)(mx >> 7);          // biased exponent of the maximum (0 for zero / subnormal rows)
        if (eb < 1) eb = 1;
        const int e = (eb - 127) - 13;    // x * 2^-e has its maximum in [2^13, 2^14)
        // 2^-e as one or two float factors (|e| can reach 139, beyond one float exponent)
        const float down = e > 0 ? __uint_as_float((uint32_t)(127 - min(e, 126)) << 23) : __uint_as_float((uint32_t)(127 + min(-e, 127)) << 23);
        const float down2 = e < -127 ? __uint_as_float((uint32_t)(127 + (-e - 127)) << 23) : 1.f;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const int v = c * 256 + threadIdx.x;
            if (v < nv) dst[v] = to_f16_scaled(keep[c], down, down2);
        }
        if (threadIdx.x == 0) xscale[slot] = ldexpf(1.f, e);
    }
}

}  // namespace

// (32 entries more: the epilogue warps read the row scales in blocks of 32)
size_t prefill_scratch_bytes(int M, int K) { return round_up((size_t)M * K * 2, 256) + round_up((size_t)M * 4 + 128, 256); }

dmr_status_t launch_prefill(const uint16_t *X, int M, RowSel sel, const void *qweight, const uint16_t *scales,
                            const uint8_t *zeros, int N, int K, int bits, int g, void *Y, dmr_out_t out,
                            void *scratch, float *partial, int32_t *status, cudaStream_t st) {
    const int sms = device_sm_count();
    // activations: gather (routed calls), rescale each row by a power of two and convert to fp16
    uint16_t *Xh = reinterpret_cast<uint16_t *>(scratch);
    float *xscale = reinterpret_cast<float *>(reinterpret_cast<char *>(scratch) + round_up((size_t)M * K * 2, 256));
    {
        const int blocks = M < sms * 16 ? M : sms * 16;
        cudaError_t e;
        if (K <= 2 * 2048) e = launch_pdl(xprep_kernel<2>, dim3((unsigned)blocks), dim3(256), 0, st, X, K, M, sel.idx, sel.count, Xh, xscale);
        else if (K <= 8 * 2048) e = launch_pdl(xprep_kernel<8>, dim3((unsigned)blocks), dim3(256), 0, st, X, K, M, sel.idx, sel.count, Xh, xscale);
        else if (K <= 16 * 2048) e = launch_pdl(xprep_kernel<16>, dim3((unsigned)blocks), dim3(256), 0, st, X, K, M, sel.idx, sel.count, Xh, xscale);
        else return DMR_ERR_UNSUPPORTED;
        if (e != cudaSuccess) {
            g_last_cuda_error = (int)e;
            (void)cudaGetLastError();
            return DMR_ERR_CUDA;
        }
        dmr_status_t r = check_launch();
        if (r != DMR_OK) return r;
    }
    return launch_pair(Xh, M, sel, xscale, qweight, scales, zeros, N, K, bits, g, Y, out, partial, status, st);
}

}  // namespace dmr
