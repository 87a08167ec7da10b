// Packed codes -> fp16 operand rows: what the tensor-core kernels' unpack threads do with one feature row and k block.
#pragma once

#include "sm100.cuh"

namespace dmr {

#ifdef __CUDACC__
// Largest magnitude pattern among a feature's G bf16 scales (sign bit cleared): eight scales per 16-byte load when the
// row of the table allows it, so that a work item's set-up is a handful of independent loads, not a chain of G.
__device__ __forceinline__ uint32_t scale_row_max(const uint16_t *sp, int G) {
    uint32_t m0 = 0, m1 = 0;
    int gi = 0;
    // scalar loads up to the first 16-byte boundary, 16-byte loads over the aligned middle, scalar loads for the rest
    const int head = (int)(((16u - (uint32_t)(reinterpret_cast<uintptr_t>(sp) & 15u)) & 15u) >> 1);
    for (; gi < G && gi < head; ++gi) m0 = max(m0, (uint32_t)__ldg(sp + gi) & 0x7FFFu);
    for (; gi + 8 <= G; gi += 8) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(sp + gi));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            m0 = max(m0, w[i] & 0x7FFFu);
            m1 = max(m1, (w[i] >> 16) & 0x7FFFu);
        }
    }
    for (; gi < G; ++gi) m1 = max(m1, (uint32_t)__ldg(sp + gi) & 0x7FFFu);
    return max(m0, m1);
}

// The power of two of a feature's largest scale, and its inverse: the unpack threads multiply the scales with the inverse (s' in
// (0, 2)), the epilogue with the power itself.
__device__ __forceinline__ int feature_exponent(const uint16_t *sp, int G) {
    const int fb = (int)(scale_row_max(sp, G) >> 7);
    return fb < 1 ? 1 : (fb > 253 ? 253 : fb);
}
__device__ __forceinline__ float feature_scale(const uint16_t *sp, int G) { return __uint_as_float((uint32_t)feature_exponent(sp, G) << 23); }

// One thread's feature row: codes, scales and zero points of a k block of 64 turned into the weights s' (q - zero) - the exact integer
// q - zero, then ONE rounding of the product to fp16 - as one 128-byte row of a swizzled K-major tile.
template <int BITS>
struct UnpackRow {
    const uint16_t *sp;
    const uint8_t *zp;
    const uint32_t *wrow;  // 3-bit codes: the row's words in global memory, or nullptr if the caller sets the words of each k block
    float fdown;
    uint32_t sb, zb, sb_next, zb_next;
    uint2 w3a, w3b, w3c, n3a, n3b, n3c;

    __device__ __forceinline__ void begin(const uint16_t *sp_, const uint8_t *zp_, int G, const uint32_t *wrow_) {
        sp = sp_;
        zp = zp_;
        wrow = wrow_;
        fdown = __uint_as_float((uint32_t)(254 - feature_exponent(sp, G)) << 23);
        sb_next = zb_next = 0;
        n3a = n3b = n3c = make_uint2(0u, 0u);
    }
    // Requests scale, zero point (and 3-bit words) of a k block; take() makes them the current ones.
    __device__ __forceinline__ void fetch(int kb, int grp) {
        sb_next = __ldg(sp + grp);
        zb_next = __ldg(zp + grp);
        if (BITS == 3 && wrow) {
            n3a = __ldg(reinterpret_cast<const uint2 *>(wrow + kb * 6));
            n3b = __ldg(reinterpret_cast<const uint2 *>(wrow + kb * 6 + 2));
            n3c = __ldg(reinterpret_cast<const uint2 *>(wrow + kb * 6 + 4));
        }
    }
    __device__ __forceinline__ void take() {
        sb = sb_next;
        zb = zb_next;
        w3a = n3a;
        w3b = n3b;
        w3c = n3c;
    }
    __device__ __forceinline__ void set_words(uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f) {
        w3a = make_uint2(a, b);
        w3b = make_uint2(c, d);
        w3c = make_uint2(e, f);
    }
    // src: the row's packed codes in shared memory; dst: its 128 bytes of the tile; r: the row's number in the tile.
    __device__ __forceinline__ void unpack(uint32_t src, uint32_t dst, int r) const {
        constexpr int CH = 8, c_lo = 0;  // 16-byte chunks (8 weights each)
        const uint32_t swz = (uint32_t)(r & 7);
        if constexpr (BITS == 3) {
            // fp16 patterns: a half-word holds five codes at bits 0, 3, 6, 9, 12.  0x6400 | (bits 0..2) = 1024 + q,
            // 0x6400 | (bits 3..5) = 1024 + 8 q, 0x6400 | (bits 6..8) = 1024 + 64 q without a shift (10 mantissa
            // bits); one shift by 9 brings the last two down.  Minus the matching 1024 + zero is exact, then one
            // rounding of the product with s', s'/8 or s'/64.
            const float sf = __uint_as_float(sb << 16) * fdown;
            uint32_t s2, s2_8, s2_64;
            asm("cvt.rn.f16x2.f32 %0, %1, %1;" : "=r"(s2) : "f"(sf));
            asm("cvt.rn.f16x2.f32 %0, %1, %1;" : "=r"(s2_8) : "f"(sf * 0.125f));
            asm("cvt.rn.f16x2.f32 %0, %1, %1;" : "=r"(s2_64) : "f"(sf * 0.015625f));
            const uint32_t z1 = 0x6400u | zb, z8 = 0x6400u | (zb << 3), z64 = 0x6400u | (zb << 6);
            const uint32_t zo1 = z1 | (z1 << 16), zo8 = z8 | (z8 << 16), zo64 = z64 | (z64 << 16);
            const uint32_t words[6] = {w3a.x, w3a.y, w3b.x, w3b.y, w3c.x, w3c.y};
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {  // 32 codes = three words = four 16-byte chunks of fp16 weights
                uint32_t D[16];  // pair 5 j + i = codes (10 j + i, 10 j + 5 + i); pair 15 = codes (30, 31)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const uint32_t u = words[3 * blk + j], u9 = u >> 9;
                    D[5 * j + 0] = f16x2_mul(f16x2_sub(lop3_and_or(u, 0x00070007u, 0x64006400u), zo1), s2);
                    D[5 * j + 1] = f16x2_mul(f16x2_sub(lop3_and_or(u, 0x00380038u, 0x64006400u), zo8), s2_8);
                    D[5 * j + 2] = f16x2_mul(f16x2_sub(lop3_and_or(u, 0x01C001C0u, 0x64006400u), zo64), s2_64);
                    D[5 * j + 3] = f16x2_mul(f16x2_sub(lop3_and_or(u9, 0x00070007u, 0x64006400u), zo1), s2);
                    D[5 * j + 4] = f16x2_mul(f16x2_sub(lop3_and_or(u9, 0x00380038u, 0x64006400u), zo8), s2_8);
                }
                {
                    uint32_t t = lop3_and_or(words[3 * blk] >> 15, 0x00010001u, 0x64006400u);
                    t = lop3_and_or(words[3 * blk + 1] >> 14, 0x00020002u, t);
                    t = lop3_and_or(words[3 * blk + 2] >> 13, 0x00040004u, t);
                    D[15] = f16x2_mul(f16x2_sub(t, zo1), s2);
                }
                // code a of the block: pair and half it sits in; the tile wants neighbours (2 v, 2 v + 1) side by side
                auto pair_of = [](int a) { return a >= 30 ? 15 : 5 * (a / 10) + (a % 10) % 5; };
                auto high_of = [](int a) { return a >= 30 ? a - 30 : ((a % 10) >= 5 ? 1 : 0); };
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) {
                    uint32_t o[4];
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) {
                        const int a0 = 8 * c4 + 2 * v4, a1 = a0 + 1;
                        o[v4] = prmt(D[pair_of(a0)], D[pair_of(a1)], (high_of(a1) ? 0x7600u : 0x5400u) | (high_of(a0) ? 0x32u : 0x10u));
                    }
                    const uint32_t addr = dst + ((((uint32_t)(4 * blk + c4)) ^ swz) << 4);
                    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]) : "memory");
                }
            }
        } else if constexpr (BITS == 4) {
            uint32_t w[CH];
#pragma unroll
            for (int c4 = 0; c4 < CH; c4 += 4)
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(w[c4]), "=r"(w[c4 + 1]), "=r"(w[c4 + 2]), "=r"(w[c4 + 3])
                             : "r"(src + 4 * (c_lo + c4)));
            // fp16 patterns: 0x6400 | q = 1024 + q and 0x6400 | (q << 4) = 1024 + 16 q (no shift needed
            // for the odd codes); minus 1024 + zero (or 1024 + 16 zero) is exact; then one rounding
            const float sf = __uint_as_float(sb << 16) * fdown;
            uint32_t s2, s2_16;
            asm("cvt.rn.f16x2.f32 %0, %1, %1;" : "=r"(s2) : "f"(sf));
            asm("cvt.rn.f16x2.f32 %0, %1, %1;" : "=r"(s2_16) : "f"(sf * 0.0625f));
            const uint32_t zz = 0x6400u | zb, zz16 = 0x6400u | (zb << 4);
            const uint32_t zoff = zz | (zz << 16), zoff16 = zz16 | (zz16 << 16);
#pragma unroll
            for (int cc = 0; cc < CH; ++cc) {  // word c = codes 8c .. 8c+7 = 16-byte chunk c of the row
                const int c = c_lo + cc;
                const uint32_t w8 = w[cc] >> 8;
                const uint32_t d04 = f16x2_mul(f16x2_sub(lop3_and_or(w[cc], 0x000F000Fu, 0x64006400u), zoff), s2);
                const uint32_t d15 = f16x2_mul(f16x2_sub(lop3_and_or(w[cc], 0x00F000F0u, 0x64006400u), zoff16), s2_16);
                const uint32_t d26 = f16x2_mul(f16x2_sub(lop3_and_or(w8, 0x000F000Fu, 0x64006400u), zoff), s2);
                const uint32_t d37 = f16x2_mul(f16x2_sub(lop3_and_or(w8, 0x00F000F0u, 0x64006400u), zoff16), s2_16);
                const uint32_t o01 = prmt(d04, d15, 0x5410), o45 = prmt(d04, d15, 0x7632);
                const uint32_t o23 = prmt(d26, d37, 0x5410), o67 = prmt(d26, d37, 0x7632);
                const uint32_t addr = dst + ((((uint32_t)c) ^ swz) << 4);
                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(o01), "r"(o23), "r"(o45), "r"(o67) : "memory");
            }
        } else {
            const float zf = __uint_as_float(0x4B000000u | zb);  // 2^23 + zero
            const float sf = __uint_as_float(sb << 16) * fdown;
            // A row of codes is 64 bytes = four 16-byte pieces.  Lane r starts at piece (r / 2) % 4, so that the eight
            // lanes of a load phase read eight different bank groups (all starting at piece 0 would meet in two).
            // Piece q holds codes 16 q .. 16 q + 15 = chunks 2 q and 2 q + 1 of the fp16 row.
#pragma unroll
            for (int j = 0; j < CH / 2; ++j) {
                const uint32_t q = ((uint32_t)j + (uint32_t)(r >> 1)) & 3u;
                uint32_t wq[4];
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(wq[0]), "=r"(wq[1]), "=r"(wq[2]), "=r"(wq[3]) : "r"(src + 16u * q));
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    uint32_t o[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t u = wq[2 * e + h];
                        float f[4];
#pragma unroll
                        for (int b = 0; b < 4; ++b)  // (q - zero) exactly, times the scale exactly (8 x 8 bits)
                            f[b] = __fmul_rn(__fsub_rn(__uint_as_float(prmt(u, 0x4B000000u, 0x7650u + (uint32_t)b)), zf), sf);
                        o[2 * h] = pack_f16x2_rn(f[0], f[1]);  // the one rounding
                        o[2 * h + 1] = pack_f16x2_rn(f[2], f[3]);
                    }
                    const uint32_t addr = dst + (((2u * q + (uint32_t)e) ^ swz) << 4);
                    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(o[0]), "r"(o[1]), "r"(o[2]), "r"(o[3]) : "memory");
                }
            }
        }
    }
};
#endif  // __CUDACC__

}  // namespace dmr
