// Low-bit linear layers on the tensor cores (3-, 4- and 8-bit codes): activation preparation for all batches, and for 33 to 128 rows
// (more go to pair.cu) a persistent, warp-specialised
// tcgen05 GEMM with the dequantisation fused into the operand pipeline.  Prefill is a dense
// contraction (its cost is folded into the per-token latency, App. "Latency coefficients"), so it
// belongs on the tensor cores.
//
// Orientation: the weights are the 128-row operand (D[n][m] = sum_k W^[n][k] X[m][k]), one
// tensor-memory lane per output feature, BN (64 or 128) activation rows as the N operand.
//
// Per 64-wide k block and stage of the ring:
//   warp 0      TMA: the packed code tile [128 features x 32 or 64 bytes] and the activation tile
//               [BN rows x 128 bytes, 128-byte swizzle] land in shared memory (one mbarrier);
//   warps 2..13  one thread per feature row turns its codes into the fp16 weights s' * (q - zero)
//               (exact integer q - zero, then ONE rounding of the product to 11 significant bits)
//               and stores them as the swizzled K-major A tile;
//   warp 1      one lane issues four tcgen05.mma (128 x BN x 16) that accumulate into one of two
//               fp32 accumulators in tensor memory, and commits the stage back to the producer;
//   the last four warps
//               drain the finished accumulator of the previous tile (tcgen05.ld) into Y while the
//               next tile's MMAs run into the other accumulator (a block of 32 rows at a time: the rows' scales and
//               output rows come from one coalesced load each, never from loads inside the store loop).
// CTAs are persistent: CTA b takes tiles b, b + grid, ...  Every wait is bounded.
//
// Operand precision.  The MMA runs in fp16 x fp16 -> fp32 (kind::f16) instead of bf16: a bf16 A
// operand would round every dequantized weight to 8 significant bits (1.5e-3 rms relative error of
// the outputs, uncomfortably close to the 2e-3 acceptance bound), fp16 keeps 11 (1.8e-4).  To stay
// inside fp16's range whatever the inputs, a preparation kernel rescales every activation row by a
// power of two (row maximum into [2^13, 2^14): exact for all elements within 2^-27 of the maximum)
// and the unpack threads rescale a feature's scales by the power of two of its largest one; the
// epilogue multiplies the two powers of two back in (exact).
#include <cuda_bf16.h>

#include <type_traits>

#include "sm100.cuh"
#include "unpack.cuh"

namespace dmr {

namespace {

constexpr int PM = 128;  // features per tile (MMA M)
constexpr int PK = 64;   // k per stage

template <int BITS, int BN>
struct PrefillCfg {
    static constexpr int A_BYTES = PM * PK * 2;              // 16 KB of fp16 weights
    static constexpr int B_BYTES = BN * PK * 2;              // activations
    static constexpr int P_ROW = PK * BITS / 8;              // packed bytes per feature per stage
    static constexpr int P_BYTES = BITS == 3 ? 0 : PM * P_ROW;  // 4 or 8 KB (3-bit rows are 24 bytes per stage, which no
                                                                // TMA box can be: the unpack threads read them from global memory)
    static constexpr int STAGE = A_BYTES + B_BYTES + ((P_BYTES + 1023) / 1024) * 1024;
    static constexpr int S_RAW = (212 * 1024) / STAGE;
    static constexpr int S = S_RAW > 8 ? 8 : S_RAW;
    static constexpr int TMEM_COLS = 2 * BN;                 // two accumulators
    // unpack warps: three groups of four, group i takes every third stage of the ring (small batches: a stage's MMAs are short and the
    // unpack chain's latency is what is left)
    static constexpr int UW = 12;
    // epilogue warps: one per tensor-memory lane quadrant (eight would make the 704 threads spill)
    static constexpr int EW = 4;
    static constexpr int THREADS = 32 * (2 + UW + EW);
    static constexpr size_t SMEM = (size_t)S * STAGE + 1024 /*alignment*/ + 512 /*barriers*/;
};

struct PrefillArgs {
    const uint16_t *scales;
    const uint8_t *zeros;
    const uint32_t *qweight3;  // 3-bit codes (read by the unpack threads; 4- and 8-bit codes come through the tensor map)
    const float *xscale;   // power of two each prepared activation row was divided by
    void *Y;
    const int32_t *idx;    // routed: output row of batch slot m (nullptr = identity)
    const int32_t *count;  // routed: number of valid slots (nullptr = M)
    int32_t *status;
    int M, N, K, g_size;
    int n_tiles, m_tiles;
    // split-K (batches of one row tile on layers with few feature tiles): a work item is (tile, split); split z sums the
    // k blocks [z kb_per_split, (z + 1) kb_per_split) and writes fp32 partial sums [z][M][N] that a second kernel adds
    // up in split order.  splits == 1: the tile's whole k range, outputs written directly.
    float *partial;
    int splits, kb_per_split;
};


// Activation preparation: Xh[slot][k] = fp16(X[row(slot)][k] * 2^-e), xscale[slot] = 2^e, with e chosen
// per row so that the row's largest magnitude lands in [2^13, 2^14).  Slots past the valid count
// (routed calls) are zero-filled.  `idx` / `count` as in the GEMM (nullptr = identity).
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

// SPLITK: work items are (tile, split) and the epilogue writes fp32 partial sums; otherwise an item is a tile with its whole
// k range (a compile-time choice: the large-batch instance carries none of the split bookkeeping).
template <int BITS, int BN, bool OUT_F32, bool SPLITK>
__global__ void __launch_bounds__(PrefillCfg<BITS, BN>::THREADS, 1)
prefill_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const PrefillArgs a) {
    using Cfg = PrefillCfg<BITS, BN>;
    constexpr int S = Cfg::S;
    extern __shared__ uint8_t smem_dyn[];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
    auto a_tile = [&](int s) { return base + (uint32_t)s * Cfg::STAGE; };
    auto b_tile = [&](int s) { return base + (uint32_t)s * Cfg::STAGE + Cfg::A_BYTES; };
    auto p_tile = [&](int s) { return base + (uint32_t)s * Cfg::STAGE + Cfg::A_BYTES + Cfg::B_BYTES; };
    const uint32_t bar_base = base + (uint32_t)S * Cfg::STAGE;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 64u + 8u * s; };
    auto ready_bar = [&](int s) { return bar_base + 128u + 8u * s; };
    auto tfull_bar = [&](int b) { return bar_base + 192u + 8u * b; };
    auto tempty_bar = [&](int b) { return bar_base + 208u + 8u * b; };
    const uint32_t tmem_slot = bar_base + 224u;
    volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(base_ptr + S * Cfg::STAGE + 224);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
            mbar_init(ready_bar(s), 4);   // one arrival per warp of the group that unpacks the stage
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), Cfg::EW);  // one arrival per epilogue warp
        }
        fence_barrier_init();
        prefetch_tensor_map(&map_w);
        prefetch_tensor_map(&map_x);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, Cfg::TMEM_COLS);
        tmem_relinquish();
    }
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot_ptr;

    // Set-up done (barriers, tensor memory): only now wait for the kernels before this one - the prepared activations, the
    // routed row lists - and let the kernel behind this one (the split-K sum) start its own set-up.
    pdl_wait();
    if constexpr (SPLITK) pdl_launch_dependents();  // (a large batch's successor would only sit on the SMs and wait)
    const int nkb = a.K / PK;
    // a routed call sizes the grid for M rows but only the first `rows` slots hold anything
    const int rows = a.count ? min(*a.count, a.M) : a.M;
    const int n_splits = SPLITK ? a.splits : 1;
    const int total_tiles = a.n_tiles * ((rows + BN - 1) / BN) * n_splits;  // work items: (tile, split), split fastest
    const int G = a.K / a.g_size;
    const int kb_per_group = a.g_size / PK;  // >= 1

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            constexpr uint32_t TX = Cfg::B_BYTES + Cfg::P_BYTES;
            uint32_t it = 0;  // k blocks issued so far, over all tiles
            bool ok = true;
            for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
                const int split = SPLITK ? tile % n_splits : 0, tl = SPLITK ? tile / n_splits : tile;
                const int kb_lo = SPLITK ? split * a.kb_per_split : 0, kb_hi = SPLITK ? min(nkb, kb_lo + a.kb_per_split) : nkb;
                const int n0 = (tl % a.n_tiles) * PM, m0 = (tl / a.n_tiles) * BN;
                for (int kb = kb_lo; kb < kb_hi; ++kb, ++it) {
                    const int s = it % S;
                    if (it >= (uint32_t)S && !mbar_wait(empty_bar(s), ((it / S) - 1) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    mbar_expect_tx(full_bar(s), TX);
                    tma_load_2d(b_tile(s), &map_x, full_bar(s), kb * PK, m0);
                    if constexpr (BITS != 3) tma_load_2d(p_tile(s), &map_w, full_bar(s), kb * Cfg::P_ROW, n0);
                }
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        // The whole warp runs the loop: stage numbers, descriptors and accumulator addresses are then the same in all
        // lanes (the compiler can keep them in uniform registers, which the MMA instruction reads), and one lane issues.
        {
            constexpr uint32_t IDESC = umma_idesc_f16(PM, BN);
            // Operand descriptors: built once for stage 0; a stage and a k step only move the 14-bit address field (16-byte
            // units), so each MMA costs an add, not a descriptor's worth of dependent shifts and ORs.
            const uint64_t desc_a0 = umma_desc_sw128(a_tile(0)), desc_b0 = umma_desc_sw128(b_tile(0));
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
            uint32_t it = 0, tile_it = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x, ++tile_it) {
                const int buf = tile_it & 1;
                // the epilogue must have drained this accumulator (used two tiles ago)
                if (tile_it >= 2 && !mbar_wait(tempty_bar(buf), ((tile_it >> 1) - 1) & 1, a.status)) break;
                tcgen05_fence_after();
                const uint32_t d_tmem = tmem_u + (uint32_t)(buf * BN);
                const int kb_lo = SPLITK ? (tile % n_splits) * a.kb_per_split : 0, kb_hi = SPLITK ? min(nkb, kb_lo + a.kb_per_split) : nkb;
                for (int kb = kb_lo; kb < kb_hi; ++kb, ++it) {
                    const int s = it % S;
                    if (!mbar_wait(ready_bar(s), (it / S) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    tcgen05_fence_after();
                    const uint64_t stage_off = (uint64_t)(((uint32_t)s * (uint32_t)Cfg::STAGE) >> 4);
                    const uint64_t desc_a = desc_a0 + stage_off, desc_b = desc_b0 + stage_off;
                    if (lane == 0) {
#pragma unroll
                        for (int j = 0; j < PK / 16; ++j)  // 16 k values = 32 bytes of a row = two 16-byte units
                            umma_bf16_ss(d_tmem, desc_a + (uint64_t)(2 * j), desc_b + (uint64_t)(2 * j), IDESC,
                                         (kb == kb_lo && j == 0) ? 0u : 1u);
                        umma_commit(empty_bar(s));
                    }
                    __syncwarp();
                }
                if (ok && lane == 0) umma_commit(tfull_bar(buf));
                __syncwarp();
            }
        }
    } else if (warp < 2 + Cfg::UW) {
        // ================= unpack warps: codes -> fp16 weights s' * (q - zero) =================
        // A stage's chain (wait, load, convert, store, fence, arrive) is a string of shared-memory round trips that
        // one group of four warps cannot overlap with itself, so NG groups work on different stages of the ring
        // at the same time: group i takes the stages whose running number is i modulo NG.
        const int r = ((warp - 2) & 3) * 32 + lane;  // feature row of the tile
        constexpr int NG = Cfg::UW / 4;
        const int grp_id = (warp - 2) >> 2;
        uint32_t it0 = 0;  // running number of the work item's first stage
        bool ok = true;
        for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
            const int split = SPLITK ? tile % n_splits : 0, tl = SPLITK ? tile / n_splits : tile;
            const int kb_lo = SPLITK ? split * a.kb_per_split : 0, kb_hi = SPLITK ? min(nkb, kb_lo + a.kb_per_split) : nkb;
            const int n = min((tl % a.n_tiles) * PM + r, a.N - 1);
            UnpackRow<BITS> row;
            row.begin(a.scales + (size_t)n * G, a.zeros + (size_t)n * G, G, BITS == 3 ? a.qweight3 + (size_t)n * (size_t)(a.K / 32 * 3) : nullptr);
            int kb = kb_lo + (int)(((uint32_t)grp_id + (uint32_t)NG - it0 % (uint32_t)NG) % (uint32_t)NG);  // this group's first k block of the item
            if (kb < kb_hi) row.fetch(kb, kb / kb_per_group);
            for (; kb < kb_hi; kb += NG) {
                const uint32_t it = it0 + (uint32_t)(kb - kb_lo);
                const int s = it % S;
                row.take();
                // what this group's next k block needs from global memory, fetched while this block is unpacked
                if (kb + NG < kb_hi) row.fetch(kb + NG, (kb + NG) / kb_per_group);
                if (!mbar_wait(full_bar(s), (it / S) & 1, a.status)) {
                    ok = false;
                    break;
                }
                row.unpack(p_tile(s) + r * Cfg::P_ROW, a_tile(s) + r * 128, r);
                fence_proxy_async_smem();  // the tile must be visible to the tensor core's reads
                __syncwarp();
                if (lane == 0) mbar_arrive(ready_bar(s));
            }
            it0 += (uint32_t)(kb_hi - kb_lo);
        }
    } else {
        // ================= epilogue warps =================
        const int q = warp & 3;        // tensor-memory lane quadrant this warp may read
        constexpr int CW = BN / (Cfg::EW / 4);                   // columns (batch slots) of a tile this warp drains
        const int c_begin = ((warp - 2 - Cfg::UW) >> 2) * CW;
        const int r = q * 32 + lane;   // feature row of the tile
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        uint32_t tile_it = 0;
        for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x, ++tile_it) {
            const int buf = tile_it & 1;
            const int split = SPLITK ? tile % n_splits : 0, tl = SPLITK ? tile / n_splits : tile;
            const int n = (tl % a.n_tiles) * PM + r, m0 = (tl / a.n_tiles) * BN;
            // the power of two the unpack threads divided this feature's scales by, undone here
            const float fscale = feature_scale(a.scales + (size_t)min(n, a.N - 1) * G, G);
            if (!mbar_wait(tfull_bar(buf), (tile_it >> 1) & 1, a.status)) break;
            tcgen05_fence_after();
#pragma unroll 1
            for (int c0 = c_begin; c0 < c_begin + CW; c0 += 32) {
                uint32_t u[32];
                tmem_ld_x16(lane_addr + (uint32_t)(buf * BN + c0), *reinterpret_cast<uint32_t(*)[16]>(&u[0]));
                tmem_ld_x16(lane_addr + (uint32_t)(buf * BN + c0 + 16), *reinterpret_cast<uint32_t(*)[16]>(&u[16]));
                tmem_ld_wait();
                if (c0 + 32 >= c_begin + CW) {  // this warp's share of the accumulator is in registers: hand it back
                    tcgen05_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty_bar(buf));
                }
                // Row scales of this block of 32 batch slots: eight 16-byte loads from one address for the whole warp (the table
                // is padded to a multiple of 64 entries).  A load per element inside the guarded loop below would be a chain of
                // 32 exposed round trips, and every shuffle or load is one more instruction through the memory pipe, which the
                // operand tiles keep busy.  Output rows of a routed call: one coalesced load, handed round by shuffles.
                float xs[32];
                {
                    const float4 *xp = reinterpret_cast<const float4 *>(a.xscale + m0 + c0);
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4) {
                        const float4 t = __ldg(xp + q4);
                        xs[4 * q4] = t.x;
                        xs[4 * q4 + 1] = t.y;
                        xs[4 * q4 + 2] = t.z;
                        xs[4 * q4 + 3] = t.w;
                    }
                }
                const bool listed = !SPLITK && a.idx != nullptr;
                const int m_lane = m0 + c0 + lane;
                const int row_lane = (listed && m_lane < rows) ? a.idx[m_lane] : m_lane;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const int m = m0 + c0 + c;
                    const int row = listed ? __shfl_sync(0xffffffffu, row_lane, c) : m;
                    if (n < a.N && m < rows) {
                        const float v = (__uint_as_float(u[c]) * xs[c]) * fscale;
                        if constexpr (SPLITK) {  // this split's share, by batch slot; the reduction scatters the rows
                            a.partial[((size_t)split * a.M + m) * a.N + n] = v;
                        } else {
                            if (OUT_F32) reinterpret_cast<float *>(a.Y)[(size_t)row * a.N + n] = v;
                            else reinterpret_cast<__nv_bfloat16 *>(a.Y)[(size_t)row * a.N + n] = __float2bfloat16_rn(v);
                        }
                    }
                }
            }
        }
    }

    // ---- teardown: every role's loop is bounded, so all warps arrive here ----
    tcgen05_fence_before();
    __syncthreads();
    if (warp == 1) {
        tcgen05_fence_after();
        tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
    }
}

template <int BITS, int BN>
dmr_status_t launch_prefill_t(const CUtensorMap &map_w, const CUtensorMap &map_x, const PrefillArgs &a, int grid,
                              dmr_out_t out, cudaStream_t st) {
    using Cfg = PrefillCfg<BITS, BN>;
    auto launch = [&](auto kernel) -> dmr_status_t {
        if (!ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), Cfg::SMEM)) return DMR_ERR_CUDA;
        cudaError_t e = launch_pdl(kernel, dim3((unsigned)grid), dim3(Cfg::THREADS), Cfg::SMEM, st, map_w, map_x, a);
        if (e != cudaSuccess) {
            g_last_cuda_error = (int)e;
            (void)cudaGetLastError();
            return DMR_ERR_CUDA;
        }
        return check_launch();
    };
    if (a.splits > 1) return launch(prefill_kernel<BITS, BN, true, true>);  // partial sums are fp32 whatever the output
    if (out == DMR_OUT_F32) return launch(prefill_kernel<BITS, BN, true, false>);
    return launch(prefill_kernel<BITS, BN, false, false>);
}

// Activation rows per tile: the smaller the activation tile, the more stages are in flight.
int prefill_bn(int M) { return M <= 64 ? 64 : 128; }

}  // namespace

bool prefill_supported(int M, int N, int K, int bits, int g) {
    if (!((bits == 3 || bits == 4 || bits == 8) && K % PK == 0 && g % PK == 0 && K <= 32768)) return false;
    if (M > 128 || bits == 3) return M > 32;  // 3-bit codes have no other tensor-core kernel
    // one tile of rows: layers with at least 16 feature tiles (split along k when the tiles alone leave SMs idle); the
    // narrow ones (k and v projections) are faster on the split-K kernel with the exact-integer operand
    return M > 32 && (N + PM - 1) / PM >= 16;
}

// Split-K factor: for layers whose tiles leave SMs idle.  As many splits as give every SM at most one work item, each
// with at least sixteen k blocks.  Depends on (M, N, K) only.
static int prefill_splits(int M, int N, int K, int sms, int *kb_per_split) {
    const int nkb = K / PK, bn = prefill_bn(M), tiles = (N + PM - 1) / PM * ((M + bn - 1) / bn);
    int splits = 1;
    if (tiles < sms) {
        splits = sms / tiles;
        if (splits > nkb / 16) splits = nkb / 16;  // a work item pays for its set-up (the feature's scale range) once
        if (splits < 1) splits = 1;
    }
    *kb_per_split = (nkb + splits - 1) / splits;
    return (nkb + *kb_per_split - 1) / *kb_per_split;  // no empty split
}

size_t prefill_partial_bytes(int M, int N, int K, int bits, int g) {
    if (pair_supported(M, N, K, bits, g)) return pair_plan(M, N, K, bits).partial_bytes;
    int kbps;
    const int splits = prefill_splits(M, N, K, device_sm_count(), &kbps);
    return splits > 1 ? (size_t)splits * M * N * sizeof(float) : 0;
}

void prefill_plan(int M, int N, int K, int *bn, int *splits, long long *tiles, int *ctas) {
    const int sms = device_sm_count();
    int kbps;
    *bn = prefill_bn(M);
    *splits = prefill_splits(M, N, K, sms, &kbps);
    *tiles = (long long)((N + PM - 1) / PM) * ((M + *bn - 1) / *bn);
    const long long items = *tiles * *splits;
    *ctas = (int)(items < sms ? items : sms);
}

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
    if (pair_supported(M, N, K, bits, g)) return launch_pair(Xh, M, sel, xscale, qweight, scales, zeros, N, K, bits, g, Y, out, partial, status, st);
    const int bn = prefill_bn(M);
    int kb_per_split;
    const int splits = prefill_splits(M, N, K, sms, &kb_per_split);
    if (splits > 1 && !partial) return DMR_ERR_WORKSPACE;
    CUtensorMap map_w, map_x;
    if (!make_tensor_map_2d(&map_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, Xh, (uint64_t)M, (uint64_t)K, (uint64_t)K * 2,
                            (uint32_t)bn, PK, TmaSwizzle::k128B))
        return DMR_ERR_CUDA;
    const uint64_t row_bytes = (uint64_t)K * bits / 8;
    if (bits == 3) {
        map_w = map_x;  // not used: a stage of 3-bit codes is 24 bytes per row, the unpack threads load it themselves
    } else if (!make_tensor_map_2d(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, qweight, (uint64_t)N, row_bytes, row_bytes, PM,
                                   (uint32_t)(PK * bits / 8), TmaSwizzle::kNone)) {
        return DMR_ERR_CUDA;
    }
    PrefillArgs a;
    a.scales = scales;
    a.zeros = zeros;
    a.qweight3 = reinterpret_cast<const uint32_t *>(qweight);
    a.xscale = xscale;
    a.Y = Y;
    a.idx = sel.idx;
    a.count = sel.count;
    a.status = status;
    a.M = M;
    a.N = N;
    a.K = K;
    a.g_size = g;
    a.n_tiles = (N + PM - 1) / PM;
    a.m_tiles = (M + bn - 1) / bn;
    a.splits = splits;
    a.kb_per_split = kb_per_split;
    a.partial = splits > 1 ? partial : nullptr;
    const long long tiles = (long long)a.n_tiles * a.m_tiles * splits;
    const int grid = (int)(tiles < sms ? tiles : sms);
    dmr_status_t r;
    auto by_rows = [&](auto bits_tag) -> dmr_status_t {
        constexpr int B = decltype(bits_tag)::value;
        if (bn == 128) return launch_prefill_t<B, 128>(map_w, map_x, a, grid, out, st);
        return launch_prefill_t<B, 64>(map_w, map_x, a, grid, out, st);
    };
    if (bits == 3) r = by_rows(std::integral_constant<int, 3>{});
    else if (bits == 4) r = by_rows(std::integral_constant<int, 4>{});
    else r = by_rows(std::integral_constant<int, 8>{});
    if (r != DMR_OK || splits == 1) return r;
    return launch_splitk_reduce(partial, splits, M, N, sel, Y, out, st);
}

}  // namespace dmr
