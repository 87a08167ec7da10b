// Weight packer: bf16 weights -> packed unsigned codes (3, 4 or 8 bits) + per-group bf16 scale and u8 zero point,
// and the matching dequantizer (test utility).
//
// The low-precision model is weight-only quantization of the decoder Linear layers with 16-bit
// activations (Sec. 5 "Experimental Models and Precision", App. "Quantization Detail").  The rule
// implemented is asymmetric min/max round-to-nearest, defined in binary64 so that the integer
// decisions (zero point, codes) do not depend on a working precision (what fp32 may stand in for is shown below):
//   lo = min(0, min w), hi = max(0, max w), s = bf16_rne((hi - lo) / qmax), zero = rint(-lo / s),
//   code = clamp(rint(w / s) + zero, 0, qmax).
#include "common.cuh"

namespace dmr {

namespace {

__device__ __forceinline__ float bf16_bits_to_float(uint32_t b) { return __uint_as_float(b << 16); }

// Nearest bf16 (ties to even) of a positive finite double, never below the smallest normal.
__device__ __forceinline__ uint32_t scale_to_bf16(double x) {
    unsigned long long u = (unsigned long long)__double_as_longlong(x);
    int e = (int)((u >> 52) & 0x7FFull) - 1023 + 127;   // bf16 biased exponent
    if (e <= 0) return 0x0080u;                          // below 2^-126: use 2^-126
    unsigned long long man = u & ((1ull << 52) - 1);
    uint32_t m7 = (uint32_t)(man >> 45);
    unsigned long long rem = man & ((1ull << 45) - 1);
    uint32_t r = ((uint32_t)e << 7) | m7;
    const unsigned long long half = 1ull << 44;
    if (rem > half || (rem == half && (m7 & 1u))) ++r;   // a carry moves into the exponent
    return r;
}

// ---- the codes in fp32 --------------------------------------------------------------------------------------------------
// A weight x and a scale s are bf16 (X 2^a and S 2^b with |X| < 256, 128 <= S < 256), so x / s is either exactly a
// half-integer or at least 1/512 away from every one: for a >= b - 1 the difference x - s h (h a half-integer) is a multiple of
// 2^(b-1), more than s / 512; for a < b - 1, |x| / s <= 255 / (4 S) <= 1/2 - 1/512.  fp32's fma(x, 1/s, 12288) rounds the
// quotient (at most 257 in magnitude; the reciprocal's error moves it by less than 2^-14) to the nearest multiple of 2^-10:
// the half-integer itself in the first case, a value on the quotient's side of it in the second.  Rounding that value to an
// integer, ties to even, therefore gives the integer the binary64 rule gives, for two fp32 instructions per weight.  The second
// addition also brings in the even part of the zero point (an even number leaves the parity of a tie alone).  A scale of 0 stands
// for "the group is not finite".
struct GroupCode {
    float rs;       // 1 / scale
    float shift;    // 1.5 2^23 - 12288 + (zero with its lowest bit cleared) + 2
    uint32_t bias;  // 2 - (zero & 1), in both half-words: what `shift` leaves on a code
};
constexpr float kGrid = 12288.f;      // 1.5 2^13: one unit in the last place is 2^-10
constexpr float kToInt = 12570624.f;  // 1.5 2^23 - kGrid

__device__ __forceinline__ GroupCode group_code(float rs, uint32_t zero) {
    GroupCode c;
    c.rs = rs;
    c.shift = kToInt + (float)((zero & ~1u) + 2u);
    c.bias = (2u - (zero & 1u)) * 0x00010001u;
    return c;
}
// rint(x / s) of a non-negative x, by the rule above.
__device__ __forceinline__ uint32_t rint_quotient(float x, float rs) {
    return __float_as_uint(__fadd_rn(__fmaf_rn(x, rs, kGrid), kToInt)) & 0xFFFFu;
}

// Two weights (fp32 bit patterns) -> their codes + bias in the two half-words.
template <int BITS>
__device__ __forceinline__ uint32_t code_pair(uint32_t x0, uint32_t x1, const GroupCode &c) {
    const uint32_t v0 = __float_as_uint(__fadd_rn(__fmaf_rn(__uint_as_float(x0), c.rs, kGrid), c.shift));
    const uint32_t v1 = __float_as_uint(__fadd_rn(__fmaf_rn(__uint_as_float(x1), c.rs, kGrid), c.shift));
    uint32_t v = __byte_perm(v0, v1, 0x5410);  // both at least 0: code + bias before the clamp
    const uint32_t top = c.bias + (uint32_t)((1 << BITS) - 1) * 0x00010001u;
    asm("min.u16x2 %0, %0, %1;" : "+r"(v) : "r"(top));
    // x >= lo and zero = rint(-lo / s) keep the code at or above 0; only the 8-bit zero point can itself have been clamped
    if (BITS == 8) asm("max.u16x2 %0, %0, %1;" : "+r"(v) : "r"(c.bias));
    return v;
}

// Eight consecutive weights -> one 4-bit word (also for 3-bit codes, before they are squeezed together).
template <int BITS>
__device__ __forceinline__ uint32_t code_nibbles(const uint4 &w, const GroupCode &c) {
    const uint32_t p0 = code_pair<BITS>(w.x << 16, w.z << 16, c);                  // codes 0, 4
    const uint32_t p1 = code_pair<BITS>(w.x & 0xFFFF0000u, w.z & 0xFFFF0000u, c);  // codes 1, 5
    const uint32_t p2 = code_pair<BITS>(w.y << 16, w.w << 16, c);
    const uint32_t p3 = code_pair<BITS>(w.y & 0xFFFF0000u, w.w & 0xFFFF0000u, c);
    return p0 + 16u * p1 + 256u * p2 + 4096u * p3 - 0x1111u * c.bias;  // a carry out of the lower half goes back with the biases
}
__device__ __forceinline__ uint2 code_bytes(const uint4 &w, const GroupCode &c) {
    const uint32_t p0 = code_pair<8>(w.x << 16, w.y << 16, c), p1 = code_pair<8>(w.x & 0xFFFF0000u, w.y & 0xFFFF0000u, c);
    const uint32_t p2 = code_pair<8>(w.z << 16, w.w << 16, c), p3 = code_pair<8>(w.z & 0xFFFF0000u, w.w & 0xFFFF0000u, c);
    return make_uint2(p0 + 256u * p1 - 257u * c.bias, p2 + 256u * p3 - 257u * c.bias);
}

// The five low nibbles of x, three bits each.
__device__ __forceinline__ uint32_t squeeze5(uint32_t x) {
    return (x & 0x7u) | ((x >> 1) & 0x38u) | ((x >> 2) & 0x1C0u) | ((x >> 3) & 0xE00u) | ((x >> 4) & 0x7000u);
}
// 3-bit codes: four neighbouring lanes hold the nibble words of one block of 32 codes; lanes 0..2 of the four return the block's
// three words (code i < 30 in word i / 10, five codes per half-word; the bits of codes 30 and 31 in bits 15 and 31).
__device__ __forceinline__ uint32_t word3(uint32_t nib, int lane) {
    const int j = lane & 3;
    const uint32_t next = __shfl_sync(0xFFFFFFFFu, nib, (lane & 28) | ((j + 1) & 3));
    const uint32_t last = __shfl_sync(0xFFFFFFFFu, nib, lane | 3);
    const uint32_t c0 = __funnelshift_r(nib, next, 8 * j), c8 = next >> (8 * j);  // codes 10 j .. 10 j + 7, then the two after them
    const uint32_t lo = squeeze5(c0), hi = squeeze5(__funnelshift_r(c0, c8, 20));
    const uint32_t b30 = (last >> (24 + j)) & 1u, b31 = (last >> (28 + j)) & 1u;
    return lo | (hi << 16) | (b30 << 15) | (b31 << 31);
}

// Codes of eight weights to their place; `oct` is the number of the eight in the flattened weight matrix.
template <int BITS>
__device__ __forceinline__ void store_codes(const uint4 &w, const GroupCode &c, bool active, size_t oct, int lane, uint32_t *__restrict__ qweight) {
    if constexpr (BITS == 4) {
        const uint32_t q = code_nibbles<4>(w, c);
        if (active) qweight[oct] = q;
    } else if constexpr (BITS == 8) {
        const uint2 q = code_bytes(w, c);
        if (active) *reinterpret_cast<uint2 *>(qweight + 2 * oct) = q;
    } else {
        const uint32_t q = word3(code_nibbles<3>(w, c), lane);
        if (active && (lane & 3) < 3) qweight[(oct >> 2) * 3 + (lane & 3)] = q;
    }
}

// ---- ranges -------------------------------------------------------------------------------------------------------------
// A range is the bf16 pair {hi, -lo}, both at least 0; NaN and infinity come through (the .NaN forms of max and min).
__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t bmin2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t range_of8(const uint4 &w) {
    const uint32_t mx = bmax2(bmax2(w.x, w.y), bmax2(w.z, w.w));
    const uint32_t mn = bmin2(bmin2(w.x, w.y), bmin2(w.z, w.w)) ^ 0x80008000u;
    return bmax2(bmax2(__byte_perm(mx, mn, 0x5410), __byte_perm(mx, mn, 0x7632)), 0u);
}

// Scale, reciprocal and zero point of a range: the scale in binary64 (one division per group), the zero point like a code.
__device__ __forceinline__ void scale_of_range(uint32_t range, int qmax, uint32_t *sb_out, float *rs_out, uint32_t *zero_out) {
    const uint32_t hb = range & 0xFFFFu, lb = range >> 16;
    if ((hb & 0x7F80u) == 0x7F80u || (lb & 0x7F80u) == 0x7F80u) {
        *sb_out = 0u;
        *rs_out = 0.f;
        *zero_out = 0u;
        return;
    }
    const float hi = bf16_bits_to_float(hb & 0x7FFFu), nlo = bf16_bits_to_float(lb & 0x7FFFu);
    uint32_t sb = (hi == 0.f && nlo == 0.f) ? 0x3F80u : scale_to_bf16(__ddiv_rn(__dadd_rn((double)hi, (double)nlo), (double)qmax));
    if (sb < 0x0080u) sb = 0x0080u;
    const float rs = __fdiv_rn(1.f, bf16_bits_to_float(sb));
    *sb_out = sb;
    *rs_out = rs;
    *zero_out = min(rint_quotient(nlo, rs), (uint32_t)qmax);
}

// Groups of 32, 64, 128 or 256 weights.  Rows are whole groups, so the matrix is one flat list of groups; a warp takes
// kLoads x 256 consecutive weights, all of them requested before the first is used, 8 per lane and load, and the lanes
// of a group find its range with bf16x2 shuffles.  The scales (the only binary64 work) are computed one group per lane, all groups
// of the warp at once.  Bound by HBM (2 bytes read, 0.52 written per weight).  Four 7B linears, 4 bits, group 128 (511 MB): 1000 us with a
// binary64 division per weight, 104 us (4.9 TB/s) now.  kLoads x CTAs per SM: 4 x 5 109 us, 6 x 4 106, 8 x 2 120, 8 x 3 104, 16 x 1 144.
constexpr int kLoads = 8;
template <int BITS, int LANES /* per group: 4, 8, 16, 32 */>
__global__ void __launch_bounds__(256, 3) quantize_small_groups(const uint16_t *__restrict__ W, long long octs /* N K / 8 */,
                                                                uint32_t *__restrict__ qweight, uint16_t *__restrict__ scales,
                                                                uint8_t *__restrict__ zeros, int32_t *__restrict__ dev_status) {
    constexpr int GP = 32 / LANES;                       // groups per load
    constexpr int GROUPS = kLoads * GP;                  // groups per warp
    constexpr int ROUNDS = (GROUPS + 31) / 32;
    const int lane = threadIdx.x & 31;
    const long long oct0 = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * (kLoads * 32);
    if (oct0 >= octs) return;
    const uint4 *src = reinterpret_cast<const uint4 *>(W) + oct0 + lane;
    uint4 w[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) w[u] = oct0 + u * 32 + lane < octs ? __ldcs(src + u * 32) : make_uint4(0u, 0u, 0u, 0u);

    // lane i keeps the range of the warp's group 32 r + i
    uint32_t mine[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) mine[r] = 0u;
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
        uint32_t p = range_of8(w[u]);
#pragma unroll
        for (int o = 1; o < LANES; o <<= 1) p = bmax2(p, __shfl_xor_sync(0xFFFFFFFFu, p, o));
        const uint32_t q = LANES == 32 ? p : __shfl_sync(0xFFFFFFFFu, p, (lane % GP) * LANES);
        if (lane / GP == u % (32 / GP)) mine[u * GP / 32] = q;
    }
    float rs[ROUNDS];
    uint32_t zero[ROUNDS];
    const long long group0 = oct0 / LANES, groups = octs / LANES;
    bool bad = false;
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        uint32_t sb;
        scale_of_range(mine[r], (1 << BITS) - 1, &sb, &rs[r], &zero[r]);
        const int i = 32 * r + lane;
        if (i < GROUPS && group0 + i < groups) {
            bad |= sb == 0u;
            scales[group0 + i] = (uint16_t)sb;
            zeros[group0 + i] = (uint8_t)zero[r];
        }
    }
    if (bad && dev_status) atomicExch(dev_status, (int)DMR_ERR_NONFINITE);
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
        const int from = (u * GP) % 32 + lane / LANES;
        const GroupCode c = group_code(__shfl_sync(0xFFFFFFFFu, rs[u * GP / 32], from), __shfl_sync(0xFFFFFFFFu, zero[u * GP / 32], from));
        store_codes<BITS>(w[u], c, oct0 + u * 32 + lane < octs, (size_t)(oct0 + u * 32 + lane), lane, qweight);
    }
}

// Long groups (one group per row, up to 32768 weights): a CTA per group keeps all of it in registers, 8 vectors of 8 weights to a
// thread, so the weights are read once; small CTAs (64 threads for 4096 weights), so that an SM's other CTAs load while one of them
// is between its two barriers.  Four 7B linears, 4 bits, one group per row: 407 us with a warp per group reading it twice, 145 with
// a CTA reading it twice, 217 with CTAs of 512 threads and two vectors each, 100 now (5.1 TB/s).
constexpr int kRowVecs = 8, kRowMaxThreads = 512;
template <int BITS>
__global__ void __launch_bounds__(kRowMaxThreads, 2) quantize_row(const uint16_t *__restrict__ W, int g, uint32_t *__restrict__ qweight,
                                                                  uint16_t *__restrict__ scales, uint8_t *__restrict__ zeros,
                                                                  int32_t *__restrict__ dev_status) {
    __shared__ uint32_t part[kRowMaxThreads / 32];
    constexpr int VPT = kRowVecs;
    const int threads = (int)blockDim.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int octs = g / 8;
    const size_t oct0 = (size_t)blockIdx.x * octs;
    const uint4 *src = reinterpret_cast<const uint4 *>(W) + oct0;
    uint4 w[VPT];
#pragma unroll
    for (int u = 0; u < VPT; ++u) {
        const int c = u * threads + (int)threadIdx.x;
        w[u] = c < octs ? __ldcs(src + c) : make_uint4(0u, 0u, 0u, 0u);
    }
    uint32_t p = 0u;
#pragma unroll
    for (int u = 0; u < VPT; ++u) p = bmax2(p, range_of8(w[u]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p = bmax2(p, __shfl_xor_sync(0xFFFFFFFFu, p, o));
    if (lane == 0) part[warp] = p;
    __syncthreads();
    p = lane < threads / 32 ? part[lane] : 0u;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) p = bmax2(p, __shfl_xor_sync(0xFFFFFFFFu, p, o));
    p = __shfl_sync(0xFFFFFFFFu, p, 0);
    uint32_t sb, zero;
    float rs;
    scale_of_range(p, (1 << BITS) - 1, &sb, &rs, &zero);
    if (threadIdx.x == 0) {
        if (sb == 0u && dev_status) atomicExch(dev_status, (int)DMR_ERR_NONFINITE);
        scales[blockIdx.x] = (uint16_t)sb;
        zeros[blockIdx.x] = (uint8_t)zero;
    }
    const GroupCode gc = group_code(rs, zero);
#pragma unroll
    for (int u = 0; u < VPT; ++u) {  // every lane takes every step: 3-bit words are put together from four lanes
        const int c = u * threads + (int)threadIdx.x;
        store_codes<BITS>(w[u], gc, c < octs, oct0 + c, lane, qweight);
    }
}

// Any other group (32 to 224 weights that are no power of two, or longer than 32768): a warp per group, two passes over it (the second one comes out of the L1 or the L2).
template <int BITS>
__global__ void __launch_bounds__(256) quantize_any(const uint16_t *__restrict__ W, long long groups, int g, uint32_t *__restrict__ qweight,
                                                    uint16_t *__restrict__ scales, uint8_t *__restrict__ zeros,
                                                    int32_t *__restrict__ dev_status) {
    const int lane = threadIdx.x & 31;
    const long long item = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (item >= groups) return;
    const int octs = g / 8;
    const size_t oct0 = (size_t)item * octs;
    const uint4 *src = reinterpret_cast<const uint4 *>(W) + oct0;
    uint32_t p = 0u;
#pragma unroll 4
    for (int c = lane; c < octs; c += 32) p = bmax2(p, range_of8(__ldg(src + c)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p = bmax2(p, __shfl_xor_sync(0xFFFFFFFFu, p, o));
    uint32_t sb, zero;
    float rs;
    scale_of_range(p, (1 << BITS) - 1, &sb, &rs, &zero);
    if (lane == 0) {
        if (sb == 0u && dev_status) atomicExch(dev_status, (int)DMR_ERR_NONFINITE);
        scales[item] = (uint16_t)sb;
        zeros[item] = (uint8_t)zero;
    }
    const GroupCode gc = group_code(rs, zero);
    const int last = (octs + 31) & ~31;  // every lane takes every step: 3-bit words are put together from four lanes
#pragma unroll 4
    for (int c = lane; c < last; c += 32) {
        const bool active = c < octs;
        const uint4 w = active ? __ldg(src + c) : make_uint4(0u, 0u, 0u, 0u);
        store_codes<BITS>(w, gc, active, oct0 + c, lane, qweight);
    }
}

template <int BITS>
void quantize_bits(const uint16_t *W, int N, int K, int g, uint32_t *qweight, uint16_t *scales, uint8_t *zeros, int32_t *dev_status, cudaStream_t st) {
    const long long octs = (long long)N * K / 8, groups = (long long)N * (K / g);
    const unsigned small = (unsigned)((octs + 8 * kLoads * 32 - 1) / (8 * kLoads * 32));
    if (g == 32) quantize_small_groups<BITS, 4><<<small, 256, 0, st>>>(W, octs, qweight, scales, zeros, dev_status);
    else if (g == 64) quantize_small_groups<BITS, 8><<<small, 256, 0, st>>>(W, octs, qweight, scales, zeros, dev_status);
    else if (g == 128) quantize_small_groups<BITS, 16><<<small, 256, 0, st>>>(W, octs, qweight, scales, zeros, dev_status);
    else if (g == 256) quantize_small_groups<BITS, 32><<<small, 256, 0, st>>>(W, octs, qweight, scales, zeros, dev_status);
    else if (g > 256 && g <= 64 * kRowMaxThreads)
        quantize_row<BITS><<<(unsigned)groups, (unsigned)((g + 64 * 32 - 1) / (64 * 32) * 32), 0, st>>>(W, g, qweight, scales, zeros, dev_status);
    else quantize_any<BITS><<<(unsigned)((groups + 7) / 8), 256, 0, st>>>(W, groups, g, qweight, scales, zeros, dev_status);
}

// One thread per 8 consecutive weights of a row.
template <int BITS, bool OUT_F32>
__global__ void __launch_bounds__(256) dequantize_kernel(const uint32_t *__restrict__ qweight,
                                                         const uint16_t *__restrict__ scales,
                                                         const uint8_t *__restrict__ zeros, int N,
                                                         int K, int g, void *__restrict__ out) {
    const long long total = (long long)N * (K / 8);
    const int G = K / g;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int n = (int)(i / (K / 8));
        const int k0 = (int)(i % (K / 8)) * 8;
        const float s = bf16_bits_to_float(scales[(size_t)n * G + k0 / g]);
        const float z = (float)zeros[(size_t)n * G + k0 / g];
        uint32_t q[8];
        if (BITS == 3) {
            const uint32_t *w = qweight + (size_t)n * (K / 32 * 3) + (size_t)(k0 / 32) * 3;
            const uint32_t w0 = w[0], w1 = w[1], w2 = w[2];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = k0 % 32 + j;
                if (i < 30) {
                    const int jj = i % 10;
                    const uint32_t word = i < 10 ? w0 : (i < 20 ? w1 : w2);
                    q[j] = (word >> (jj < 5 ? 3 * jj : 16 + 3 * (jj - 5))) & 7u;
                } else {
                    const int bit = i == 30 ? 15 : 31;
                    q[j] = ((w0 >> bit) & 1u) | (((w1 >> bit) & 1u) << 1) | (((w2 >> bit) & 1u) << 2);
                }
            }
        } else if (BITS == 4) {
            uint32_t w = qweight[(size_t)n * (K / 8) + k0 / 8];
#pragma unroll
            for (int j = 0; j < 8; ++j) q[j] = (w >> (4 * j)) & 0xFu;
        } else {
            uint2 w = *reinterpret_cast<const uint2 *>(qweight + (size_t)n * (K / 4) + k0 / 4);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                q[j] = (w.x >> (8 * j)) & 0xFFu;
                q[4 + j] = (w.y >> (8 * j)) & 0xFFu;
            }
        }
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = __fmul_rn(s, (float)q[j] - z);  // exact: 8 x 9 significant bits
        if (OUT_F32) {
            float4 *o = reinterpret_cast<float4 *>((float *)out + (size_t)n * K + k0);
            o[0] = make_float4(v[0], v[1], v[2], v[3]);
            o[1] = make_float4(v[4], v[5], v[6], v[7]);
        } else {
            uint32_t p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                // round to nearest even bf16 by integer arithmetic on the fp32 pattern (values are finite)
                uint32_t a = __float_as_uint(v[2 * j]), b = __float_as_uint(v[2 * j + 1]);
                a = (a + 0x7FFFu + ((a >> 16) & 1u)) >> 16;
                b = (b + 0x7FFFu + ((b >> 16) & 1u)) >> 16;
                p[j] = a | (b << 16);
            }
            *reinterpret_cast<uint4 *>((uint16_t *)out + (size_t)n * K + k0) = make_uint4(p[0], p[1], p[2], p[3]);
        }
    }
}

}  // namespace

dmr_status_t launch_quantize(const uint16_t *W, int N, int K, int bits, int g, uint32_t *qweight,
                             uint16_t *scales, uint8_t *zeros, int32_t *dev_status, cudaStream_t st) {
    if (bits == 3) quantize_bits<3>(W, N, K, g, qweight, scales, zeros, dev_status, st);
    else if (bits == 4) quantize_bits<4>(W, N, K, g, qweight, scales, zeros, dev_status, st);
    else quantize_bits<8>(W, N, K, g, qweight, scales, zeros, dev_status, st);
    return check_launch();
}

dmr_status_t launch_dequantize(const uint32_t *qweight, const uint16_t *scales, const uint8_t *zeros,
                               int N, int K, int bits, int g, void *W_out, dmr_out_t out, cudaStream_t st) {
    const long long total = (long long)N * (K / 8);
    long long blocks = (total + 255) / 256;
    if (blocks > 148 * 64) blocks = 148 * 64;
    if (bits == 3) {
        if (out == DMR_OUT_F32)
            dequantize_kernel<3, true><<<(int)blocks, 256, 0, st>>>(qweight, scales, zeros, N, K, g, W_out);
        else
            dequantize_kernel<3, false><<<(int)blocks, 256, 0, st>>>(qweight, scales, zeros, N, K, g, W_out);
    } else if (bits == 4) {
        if (out == DMR_OUT_F32)
            dequantize_kernel<4, true><<<(int)blocks, 256, 0, st>>>(qweight, scales, zeros, N, K, g, W_out);
        else
            dequantize_kernel<4, false><<<(int)blocks, 256, 0, st>>>(qweight, scales, zeros, N, K, g, W_out);
    } else {
        if (out == DMR_OUT_F32)
            dequantize_kernel<8, true><<<(int)blocks, 256, 0, st>>>(qweight, scales, zeros, N, K, g, W_out);
        else
            dequantize_kernel<8, false><<<(int)blocks, 256, 0, st>>>(qweight, scales, zeros, N, K, g, W_out);
    }
    return check_launch();
}

}  // namespace dmr
