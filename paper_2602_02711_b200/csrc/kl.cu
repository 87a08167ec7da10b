// Step-wise KL divergence between the action distributions of the high- and the low-precision
// model: KL_t = mean over the action tokens i of step t of KL(pi_high(x_i) || pi_low(x_i)), the
// quantity the KL-ST router is trained to predict (Sec. "KL-ST Stage"; App. on search and click
// steps, definition of the per-step action-block KL).
//
// Per token, with a = high-precision logits, b = low-precision logits, p = softmax(a):
//   KL = sum_v p_v (a_v - b_v) - lse(a) + lse(b),
// formed in ONE pass over the two logit rows (2 x V elements, read once: the kernel is bound by
// memory bandwidth) with running maxima, in fp32:
//   m_a, S0 = sum e^(a - m_a), S1 = sum e^(a - m_a) (a - b);   m_b, S2 = sum e^(b - m_b)
//   KL = S1 / S0 + ((m_b - m_a) + (log S2 - log S0)).
// A vocabulary entry with p_v = 0 (a_v = -inf) contributes nothing.  A row is cut into contiguous parts (a number that
// depends on V alone), the 16-byte vectors of a part, counted from the row's start, go to a CTA's threads in turn, and the sums are
// combined in a fixed order, so the result depends neither on the grid nor on where the row lies in memory.
// A second, tiny kernel averages the tokens of each step in order.
#include <cuda_bf16.h>

#include "sm100.cuh"

namespace dmr {

namespace {

constexpr int kKlThreads = 512;
constexpr int kKlWarps = kKlThreads / 32;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
// Logits below this (-inf, a mask of the type's lowest value) are raised to it: no inf - inf anywhere, e^(x - m) is still 0.  A bf16 number whose
// product with log2 e is rounded up: where a thread has met nothing but the floor so far, the fused multiply-add of its weight leaves that
// rounding, 5e22 below zero, whose power of two is 0 (of a floor whose product is rounded down it would be infinite).
constexpr float kLogitFloor = -9.953037915854457e29f;
constexpr uint32_t kFloorPair = 0xF149F149u;  // the same as a bf16 pair

// CTAs of a cluster that share a row: the two halves of a long row end together and few tokens reach twice as many SMs (9 tokens x
// 151936: 20.5 us in one part, 18 in two; 777 tokens: 95 and 90); rows below 16384 entries would mostly pay for the exchange.
constexpr int kKlMaxParts = 2;
__host__ __device__ constexpr int kl_parts(int V) { return V >= 16384 ? 2 : 1; }
// CTAs that share a row: one for each part, except that one CTA takes a row of fp32 logits part after part (the same sums) where the halves need an
// even number of rounds of CTAs over the chip.  Whole rows fill it as well then, and a round that is nearly empty, a row's latency long, costs half
// as much of the time as they do (300 x 151936: 78 and 68 us; 444 x 99997: 91 and 68; but 250 x 151936 48 and 63, 700 x 151936 139 and 160).
// With bf16 logits, half as many bytes for the same exponentials, such a round is hidden (300 x 151936: 45 and 48 us).
inline int kl_ctas(int T, int parts, bool f32) {
    const int resident = 4 * device_sm_count();
    return f32 && parts == 2 && (T + (resident / 2 - 1)) / (resident / 2) % 2 == 0 ? 1 : parts;
}
static_assert(kKlMaxParts * kKlWarps <= 32, "the sums of a token's warps meet in one warp");

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// A thread's running sums (even and odd elements apart: two shorter chains of additions).
struct KlThread {
    float ma = -INFINITY, mb = -INFINITY;  // maxima in log2 units
    float s0[2] = {0.f, 0.f}, s1[2] = {0.f, 0.f}, s2[2] = {0.f, 0.f};
};
struct KlSums {
    float ma, s0, s1, mb, s2;
};

__device__ __forceinline__ void kl_raise(KlThread &st, float va, float vb) {
    if (va > st.ma) {
        const float r = ex2(st.ma - va);  // 0 when the old maximum was -inf
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            st.s0[i] *= r;
            st.s1[i] *= r;
        }
        st.ma = va;
    }
    if (vb > st.mb) {
        const float r = ex2(st.mb - vb);
        st.s2[0] *= r;
        st.s2[1] *= r;
        st.mb = vb;
    }
}
// One 16-byte vector of each row.  Of a, finite logits only: -inf or NaN anywhere leaves s1 not finite, which the caller looks at once per
// part of a row (kl_redo) instead of once per element; a finite one below the floor has weight 0, or leaves s1 not finite where the thread has
// met no other.
template <bool F32>
__device__ __forceinline__ void kl_vector(KlThread &st, const uint4 &qa, const uint4 &qb) {
    const uint32_t a[4] = {qa.x, qa.y, qa.z, qa.w};
    uint32_t b[4] = {qb.x, qb.y, qb.z, qb.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) b[i] = F32 ? __float_as_uint(fmaxf(__uint_as_float(b[i]), kLogitFloor)) : bmax2(b[i], kFloorPair);
    if constexpr (F32) {
        const float va = fmaxf(fmaxf(__uint_as_float(a[0]), __uint_as_float(a[1])), fmaxf(__uint_as_float(a[2]), __uint_as_float(a[3])));
        const float vb = fmaxf(fmaxf(__uint_as_float(b[0]), __uint_as_float(b[1])), fmaxf(__uint_as_float(b[2]), __uint_as_float(b[3])));
        kl_raise(st, va * kLog2e, vb * kLog2e);
    } else {
        const uint32_t ma = bmax2(bmax2(a[0], a[1]), bmax2(a[2], a[3])), mb = bmax2(bmax2(b[0], b[1]), bmax2(b[2], b[3]));
        kl_raise(st, fmaxf(lo_f(ma), hi_f(ma)) * kLog2e, fmaxf(lo_f(mb), hi_f(mb)) * kLog2e);
    }
    constexpr int N = F32 ? 4 : 8;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const float x = F32 ? __uint_as_float(a[i % 4]) : ((i & 1) ? hi_f(a[i / 2]) : lo_f(a[i / 2]));
        const float y = F32 ? __uint_as_float(b[i % 4]) : ((i & 1) ? hi_f(b[i / 2]) : lo_f(b[i / 2]));
        const float w = ex2(fmaf(x, kLog2e, -st.ma));
        st.s0[i & 1] += w;
        st.s1[i & 1] = fmaf(w, x - y, st.s1[i & 1]);
        st.s2[i & 1] += ex2(fmaf(y, kLog2e, -st.mb));
    }
}
// One element of any value: -inf, NaN and what lies below the floor count as the floor, and p_v = 0 contributes nothing whatever b_v is.
__device__ __forceinline__ void kl_element(KlThread &st, float a, float b) {
    a = fmaxf(a, kLogitFloor);
    b = fmaxf(b, kLogitFloor);
    kl_raise(st, a * kLog2e, b * kLog2e);
    const float w = ex2(fmaf(a, kLog2e, -st.ma));
    st.s0[0] += w;
    if (w > 0.f) st.s1[0] = fmaf(w, a - b, st.s1[0]);
    st.s2[0] += ex2(fmaf(b, kLog2e, -st.mb));
}

// Sixteen bytes at p, an element boundary `shift` bytes past a 16-byte one (the same for the whole row), from the two aligned
// vectors around them; the second is what the next lane loads as its first.
__device__ __forceinline__ uint4 load_shifted(const uint8_t *p, uint32_t shift) {
    const uint4 *q = reinterpret_cast<const uint4 *>(p - shift);
    if (shift == 0) return __ldcs(q);
    const uint4 v = __ldg(q), n = __ldg(q + 1);
    const bool by8 = shift & 8u, by4 = shift & 4u;
    const uint32_t t0 = by8 ? v.z : v.x, t1 = by8 ? v.w : v.y, t2 = by8 ? n.x : v.z, t3 = by8 ? n.y : v.w, t4 = by8 ? n.z : n.x,
                   t5 = by8 ? n.w : n.y;
    const uint32_t u0 = by4 ? t1 : t0, u1 = by4 ? t2 : t1, u2 = by4 ? t3 : t2, u3 = by4 ? t4 : t3, u4 = by4 ? t5 : t4;
    const uint32_t s = (shift & 2u) * 8u;
    return make_uint4(__funnelshift_r(u0, u1, s), __funnelshift_r(u1, u2, s), __funnelshift_r(u2, u3, s), __funnelshift_r(u3, u4, s));
}

// The sums of 32 lanes brought to their common maxima and added (butterfly: every lane ends with the same sums).
__device__ __forceinline__ void kl_warp_sum(KlSums &s) {
    float ma = s.ma, mb = s.mb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ma = fmaxf(ma, __shfl_xor_sync(0xFFFFFFFFu, ma, o));
        mb = fmaxf(mb, __shfl_xor_sync(0xFFFFFFFFu, mb, o));
    }
    const float ra = s.ma == ma ? 1.f : ex2(s.ma - ma), rb = s.mb == mb ? 1.f : ex2(s.mb - mb);
    s.s0 *= ra;
    s.s1 *= ra;
    s.s2 *= rb;
    s.ma = ma;
    s.mb = mb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s.s0 += __shfl_xor_sync(0xFFFFFFFFu, s.s0, o);
        s.s1 += __shfl_xor_sync(0xFFFFFFFFu, s.s1, o);
        s.s2 += __shfl_xor_sync(0xFFFFFFFFu, s.s2, o);
    }
}

template <bool F32>
__device__ __forceinline__ float kl_load(const uint8_t *row, int e) {
    if constexpr (F32) return reinterpret_cast<const float *>(row)[e];
    else return __uint_as_float((uint32_t)reinterpret_cast<const uint16_t *>(row)[e] << 16);
}
// The elements of vector v (up to the row's end) one by one from global memory.
template <bool F32>
__device__ __noinline__ KlThread kl_elements(KlThread st, const uint8_t *ra, const uint8_t *rb, int v, int V) {
    constexpr int VE = F32 ? 4 : 8;
    for (int e = v * VE; e < min(v * VE + VE, V); ++e) kl_element(st, kl_load<F32>(ra, e), kl_load<F32>(rb, e));
    return st;
}
// This thread's share of the part once more, for logits that are not finite.
template <bool F32>
__device__ __noinline__ KlThread kl_redo(const uint8_t *ra, const uint8_t *rb, int v, int end, int V) {
    KlThread st;
    for (; v < end; v += kKlThreads) st = kl_elements<F32>(st, ra, rb, v, V);
    return st;
}

// F32 = logits are fp32 (else bf16).  ALIGNED = every row starts on a 16-byte boundary.
// Bound by HBM and, with bf16 logits, as much by the two exponentials per element (16 per clock and SM: 52 us for 777 x 151936
// against 72 for the bytes).  So: 64 warps on an SM (at most 32 registers, one vector of each row in flight per thread; two in
// flight, or 48 warps, measured no better: 89 and 92 us), no test per element for logits that are not finite, bf16x2 maxima, unaligned
// rows (V not a multiple of 8) with 16-byte loads too.  777 x 151936 bf16: 106 -> 95 us (5.0 TB/s); 100 x 99997: 30 -> 21;
// 250 x 151936 fp32: 64 -> 48 (6.3 TB/s).
template <bool F32, bool ALIGNED>
__global__ void __launch_bounds__(kKlThreads, 4)
kl_token_kernel(const void *__restrict__ high, const void *__restrict__ low, int V, int parts, int ctas, float *__restrict__ kl_token) {
    constexpr int ES = F32 ? 4 : 2, VE = F32 ? 4 : 8;  // bytes per element, elements per vector
    __shared__ KlSums sums[kKlMaxParts * kKlWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = (int)(blockIdx.x % (unsigned)ctas);  // `ctas` CTAs share a row's parts: each takes one, or the only one takes all
    const size_t tok = blockIdx.x / (unsigned)ctas;
    pdl_launch_dependents();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;");  // every CTA of the cluster runs before its shared memory is written

    const size_t row = tok * V * ES;
    const uint8_t *ra = reinterpret_cast<const uint8_t *>(high) + row, *rb = reinterpret_cast<const uint8_t *>(low) + row;
    const uint32_t shift = ALIGNED ? 0u : (uint32_t)(row & 15u);  // both matrices start on 16-byte boundaries
    const int vecs = (V + VE - 1) / VE, per = (vecs + parts - 1) / parts;
    // vectors that lie, with the 16 bytes after them where those are read too, inside the row
    const int whole = shift == 0 ? V / VE : max(0, (V - VE) / VE);
#pragma unroll 1
    for (int part = rank; part < (F32 && ctas == 1 ? parts : rank + 1); ++part) {
        const int end = min(vecs, (part + 1) * per), fast = min(end, whole), first = part * per + (int)threadIdx.x;
        KlThread st;
        int v = first;
        const uint8_t *pa = ra + (size_t)v * 16, *pb = rb + (size_t)v * 16;
#pragma unroll 1
        for (; v < fast; v += kKlThreads) {
            kl_vector<F32>(st, load_shifted(pa, shift), load_shifted(pb, shift));
            pa += kKlThreads * 16;
            pb += kKlThreads * 16;
        }
        for (; v < end; v += kKlThreads) {
            // the one or two vectors at the row's end; a whole one is added like every other, whatever `shift`
            if ((v + 1) * VE > V) {
                st = kl_elements<F32>(st, ra, rb, v, V);
                continue;
            }
            uint32_t x[4], y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if constexpr (F32) {
                    x[j] = reinterpret_cast<const uint32_t *>(ra)[v * 4 + j];
                    y[j] = reinterpret_cast<const uint32_t *>(rb)[v * 4 + j];
                } else {
                    const uint16_t *p = reinterpret_cast<const uint16_t *>(ra) + v * 8 + 2 * j, *q = reinterpret_cast<const uint16_t *>(rb) + v * 8 + 2 * j;
                    x[j] = p[0] | ((uint32_t)p[1] << 16);
                    y[j] = q[0] | ((uint32_t)q[1] << 16);
                }
            }
            kl_vector<F32>(st, make_uint4(x[0], x[1], x[2], x[3]), make_uint4(y[0], y[1], y[2], y[3]));
        }
        if (!isfinite((st.s1[0] + st.s1[1]) + (st.s2[0] + st.s2[1]))) st = kl_redo<F32>(ra, rb, first, end, V);
        KlSums s;
        s.ma = st.ma;
        s.mb = st.mb;
        s.s0 = st.s0[0] + st.s0[1];
        s.s1 = st.s1[0] + st.s1[1];
        s.s2 = st.s2[0] + st.s2[1];
        kl_warp_sum(s);
        if (part == rank) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (lane < 5) {  // the warp's five numbers to the first CTA's shared memory
            const float f = lane == 0 ? s.ma : lane == 1 ? s.s0 : lane == 2 ? s.s1 : lane == 3 ? s.mb : s.s2;
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_map(smem_u32(&sums[part * kKlWarps + warp]) + 4u * lane, 0)), "f"(f) : "memory");
        }
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    if (rank != 0 || warp != 0) return;  // only the first warp of the cluster reads on
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    KlSums tot = {-INFINITY, 0.f, 0.f, -INFINITY, 0.f};
    if (lane < parts * kKlWarps) tot = sums[lane];
    kl_warp_sum(tot);
    // lse(b) - lse(a), differences first (exactly 0 for equal rows), from log2 to natural-log units
    const float dlse = ((tot.mb - tot.ma) + (log2f(tot.s2) - log2f(tot.s0))) * kLn2;
    // a row of nothing but the floor is no distribution: undefined (0 / 0) as the first one, infinitely far as the second
    if (lane == 0) kl_token[tok] = tot.s2 == 0.f && tot.s0 > 0.f ? INFINITY : tot.s1 / tot.s0 + dlse;
}

// kl_step[s] = mean of kl_token over [offsets[s], offsets[s + 1]), added in token order; 0 for an empty step.
__global__ void __launch_bounds__(128)
kl_step_kernel(const float *__restrict__ kl_token, const int32_t *__restrict__ offsets, int S, int T, float *__restrict__ kl_step) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();  // launched while the token kernel still runs
    if (s >= S) return;
    int beg = offsets[s], end = offsets[s + 1];
    beg = beg < 0 ? 0 : beg;
    end = end > T ? T : end;
    float sum = 0.f;
    for (int i = beg; i < end; ++i) sum += kl_token[i];
    kl_step[s] = end > beg ? sum / (float)(end - beg) : 0.f;
}

}  // namespace

dmr_status_t launch_stepwise_kl(const void *high, const void *low, bool f32, int T, int V, const int32_t *offsets, int S,
                                float *kl_token, float *kl_step, cudaStream_t st) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (T > 0) {
        const int parts = kl_parts(V), ctas = kl_ctas(T, parts, f32);
        const bool aligned = V % (f32 ? 4 : 8) == 0;
        auto kernel = f32 ? (aligned ? kl_token_kernel<true, true> : kl_token_kernel<true, false>)
                          : (aligned ? kl_token_kernel<false, true> : kl_token_kernel<false, false>);
        cfg.gridDim = dim3((unsigned)T * (unsigned)ctas, 1, 1);
        cfg.blockDim = dim3(kKlThreads, 1, 1);
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)ctas;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, high, low, V, parts, ctas, kl_token);
        if (e != cudaSuccess) return launch_failed(e);
        dmr_status_t r = check_launch();
        if (r != DMR_OK || S == 0) return r;
    }
    cfg.gridDim = dim3((unsigned)(S + 127) / 128, 1, 1);
    cfg.blockDim = dim3(128, 1, 1);
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kl_step_kernel, (const float *)kl_token, offsets, S, T, kl_step);
    if (e != cudaSuccess) return launch_failed(e);
    return check_launch();
}

}  // namespace dmr
