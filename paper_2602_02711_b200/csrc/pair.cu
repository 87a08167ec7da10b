// Large-batch linears (bf16 weights, or 3-, 4- and 8-bit codes) on pairs of SMs: tcgen05.mma with cta_group::2.
//
// What bounds it.  The product is a dense contraction, so the tensor cores do; what kept them waiting on one SM per tile was
// the tile's other traffic: at 128 features x 256 rows a k block of 64 takes 512 cycles of MMAs and 36 (4-bit codes) or 48 KB (bf16) of
// operands, and an SM takes in about 61 bytes a cycle from the L2 (590 and 790 cycles); shared memory moved 104 KB per k block,
// 810 cycles at 128 B a cycle.  A pair of SMs works on 256 features x up to 256 rows: each SM holds its own 128 features' weights
// and HALF of the activation rows (the tensor cores of both read both halves), so a k block costs an SM 20 or 32 KB from the L2 and
// 72 KB of shared-memory traffic, and the ring gets six or seven stages instead of four.
// Measured, four 7B linears, us, against one SM per tile: bf16 weights M = 300 240 -> 182, M = 1501 704 -> 530, M = 4096 1850 -> 1336 (1241
// TFLOP/s, 0.91 of what the card sustains under its power limit); 4-bit codes, activation preparation included, M = 400 263 -> 222,
// M = 1000 445 -> 390, M = 2048 853 -> 750, M = 4096 1680 -> 1450; 8 bits, M = 1024 576 -> 467; 3 bits, M = 1024 474 -> 389.  Three groups
// of unpack warps, or four epilogue warps, are no faster (M = 400: 237 and 235).
//
// Roles of a CTA: warp 0 copies (TMA, plain per-CTA boxes), warp 1 of the pair's first CTA issues the MMAs for both (the second CTA's
// warp 1 only passes on that its operands have landed), for codes eight warps turn them into fp16 weights (two groups that take
// alternate stages; see prefill.cu for the operand's precision), eight warps drain the accumulators (two per lane quadrant,
// alternate blocks of 32 rows) while the next tile's MMAs fill the other one.  Every wait is bounded.
//
// Tiles.  The row count of a tile is any multiple of 16 up to 256, chosen so that the rows fill the last round of tiles over the pairs
// (pair_tile_rows).  Eight row tiles are visited per feature tile before the next feature tile, so that the pairs at work share
// weights and activations in the L2.
#include <cuda_bf16.h>

#include <cmath>

#include <type_traits>

#include "sm100.cuh"
#include "unpack.cuh"

namespace dmr {

namespace {

constexpr int kPm = 128;         // features per CTA
constexpr int kPk = 64;          // k per stage
constexpr int kMaxRows = 256;    // activation rows per tile at most
constexpr int kRowGroup = 8;     // row tiles visited per feature tile

template <int BITS, bool WORDS = false>  // BITS 0: bf16 weights; WORDS: the unpack threads fetch the codes' words from global memory themselves
struct PairCfg {
    static constexpr int A_BYTES = kPm * kPk * 2;                       // 16 KB
    static constexpr int B_BYTES = kMaxRows / 2 * kPk * 2;              // 16 KB
    // Packed codes of a stage.  A k block of 3-bit codes is 24 bytes a row, which no TMA box can be: two k blocks share a box of 48
    // bytes, in a slot of its own beside the ring (S / 2 of them).  Rows of an odd number of k blocks (no multiple of 16 bytes, so that no tensor map
    // describes them) are read word by word (WORDS): 2880 x 2880, groups of 64, M = 300 / 700 / 2048 26 / 32 / 58 us (M = 300, 700 on the CUDA cores:
    // 2680, 6145); 3000 x 4544, M = 200 29.
    static constexpr bool BOX3 = BITS == 3 && !WORDS;
    static constexpr int P_ROW = BOX3 ? 48 : WORDS ? 0 : kPk * BITS / 8;
    static constexpr int P_BYTES = BITS == 0 ? 0 : kPm * P_ROW;
    static constexpr int STAGE = A_BYTES + B_BYTES + (BOX3 ? 0 : P_BYTES);
    static constexpr int S_RAW = (225 * 1024) / STAGE;
    static constexpr int S = BOX3 ? 6 : S_RAW > 8 ? 8 : S_RAW;
    // Barriers the copies of the k blocks complete on, in turn.  Where a stage comes round to the unpack groups alternately there are two per
    // stage, so that each is always waited for by the same group, phase after phase: a group that did not wait for the phase before takes
    // a parity it waits for as already there.  (An even number of stages would do too: 8-bit, 32B layer, M = 500, 4 stages for 5: 381 us
    // instead of 345; 3-bit, 7B layer, M = 1024, 4 for 6: 423 instead of 395.)
    static constexpr int F = BITS == 8 || BITS == 3 ? 2 * S : S;
    static constexpr int RING = S * STAGE + (BOX3 ? S / 2 * P_BYTES : 0);
    static constexpr int UW = BITS == 0 ? 0 : 8;                        // unpack warps
    static constexpr int EW = 8;                                        // epilogue warps
    static constexpr int THREADS = 32 * (2 + UW + EW);
    static constexpr size_t SMEM = (size_t)RING + 1024 /*alignment*/ + 512 /*barriers*/;
    static_assert(SMEM <= 227 * 1024, "stages exceed an SM's shared memory");
    static_assert(UW == 0 || F / (BOX3 ? 2 : 1) % (UW / 4) == 0, "a barrier belongs to one group of unpack warps");
    static_assert(S <= 8 && F <= 32, "room for the barriers");
};

struct PairArgs {
    const uint16_t *scales;
    const uint8_t *zeros;
    const uint32_t *words;     // 3-bit codes of rows that no tensor map describes
    const float *xscale;       // codes: power of two each prepared activation row was divided by
    void *Y;
    const int32_t *idx;        // routed: output row of batch slot m (nullptr = identity)
    const int32_t *count;      // routed: number of valid slots (nullptr = M)
    int32_t *status;
    float *partial;            // split along k: fp32 sums [splits][M][N]
    int M, N, K, g_size;
    int n_tiles, tile_rows, splits, kb_per_split;
};

// ---- cta_group::2 forms ----
__device__ __forceinline__ void tmem_alloc2(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish2() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void umma2_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// The barrier at this shared-memory offset gets one arrival in both CTAs once the MMAs issued so far have completed.
__device__ __forceinline__ void umma2_commit_both(uint32_t bar) {
    const uint16_t both = 3;
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(both) : "memory");
}

// Arrival on a barrier of either CTA of the pair.  What it announces is read by the tensor cores alone (operands: copied by TMA, or stored
// and passed through a proxy fence) or has been read (accumulators), so no memory order at cluster scope is asked for: the
// arrive.release.cluster / acquire.cluster forms cost about a microsecond a k block here (bf16, M = 4096: 3002 us against 1336).
__device__ __forceinline__ void mbar_arrive_pair(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

struct TilePos {
    int n, m, split;
};
// Work item -> tile: splits fastest, then the row tiles of a group, then feature tiles, then groups.
template <bool SPLITK>
__device__ __forceinline__ TilePos tile_pos(int item, int n_tiles, int m_tiles, int splits) {
    TilePos p;
    p.split = SPLITK ? item % splits : 0;
    const int t = SPLITK ? item / splits : item;
    const int per_group = n_tiles * kRowGroup, g = t / per_group, rem = t - g * per_group;
    const int gm = min(kRowGroup, m_tiles - g * kRowGroup);
    p.n = rem / gm;
    p.m = g * kRowGroup + rem - p.n * gm;
    return p;
}

template <int BITS, bool WORDS, bool OUT_F32, bool SPLITK>
__global__ void __launch_bounds__(PairCfg<BITS, WORDS>::THREADS, 1)
pair_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x, const PairArgs a) {
    using Cfg = PairCfg<BITS, WORDS>;
    constexpr int S = Cfg::S, F = Cfg::F;
    constexpr bool BOX3 = Cfg::BOX3;
    extern __shared__ uint8_t smem_dyn[];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)cluster_id_x(), pairs = (int)cluster_count_x();
    const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
    uint8_t *base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
    auto a_tile = [&](int s) { return base + (uint32_t)s * Cfg::STAGE; };
    auto b_tile = [&](int s) { return base + (uint32_t)s * Cfg::STAGE + Cfg::A_BYTES; };
    auto p_tile = [&](int s) {
        return BOX3 ? base + (uint32_t)(S * Cfg::STAGE + s / 2 * Cfg::P_BYTES) : base + (uint32_t)s * Cfg::STAGE + Cfg::A_BYTES + Cfg::B_BYTES;
    };
    const uint32_t bar_base = base + (uint32_t)Cfg::RING;
    auto full_bar = [&](int f) { return bar_base + 256u + 8u * f; };     // this CTA's copies have landed, k block it: f = it % F
    auto empty_bar = [&](int s) { return bar_base + 64u + 8u * s; };     // the MMAs have read the stage (both CTAs get it)
    auto ready_bar = [&](int s) { return bar_base + 128u + 8u * s; };    // first CTA: operands in place (codes: both CTAs; bf16: the second)
    auto tfull_bar = [&](int b) { return bar_base + 192u + 8u * b; };    // an accumulator is finished (both CTAs get it)
    auto tempty_bar = [&](int b) { return bar_base + 208u + 8u * b; };   // first CTA: both CTAs have drained it
    const uint32_t tmem_slot = bar_base + 224u;
    volatile uint32_t *tmem_slot_ptr = reinterpret_cast<volatile uint32_t *>(base_ptr + Cfg::RING + 224);

    if (threadIdx.x == 0) {
        for (int f = 0; f < F; ++f) mbar_init(full_bar(f), 1);
        for (int s = 0; s < S; ++s) {
            mbar_init(empty_bar(s), 1);
            mbar_init(ready_bar(s), BITS == 0 ? 1 : 8);  // codes: four unpack warps of each CTA
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), 2 * Cfg::EW);
        }
        fence_barrier_init();
        prefetch_tensor_map(&map_w);
        prefetch_tensor_map(&map_x);
    }
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers exist
    if (warp == 1) {
        tmem_alloc2(tmem_slot, 512);
        tmem_relinquish2();
    }
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot_ptr;

    pdl_wait();  // set-up done: now wait for the prepared activations, the row lists
    if constexpr (SPLITK) pdl_launch_dependents();
    const int nkb = a.K / kPk, BN = a.tile_rows;
    const int rows = a.count ? min(*a.count, a.M) : a.M;
    const int m_tiles = (rows + BN - 1) / BN;
    const int n_splits = SPLITK ? a.splits : 1;
    const int items = a.n_tiles * m_tiles * n_splits;
    auto k_lo = [&](const TilePos &p) { return SPLITK ? p.split * a.kb_per_split : 0; };
    auto k_hi = [&](const TilePos &p) { return SPLITK ? min(nkb, (p.split + 1) * a.kb_per_split) : nkb; };

    if (warp == 0) {
        // ================= copies =================
        if (lane == 0) {
            const uint32_t tx_x = (uint32_t)(BN / 2) * (kPk * 2), tx_w = BITS == 0 ? Cfg::A_BYTES : Cfg::P_BYTES;
            uint32_t it = 0;
            bool ok = true;
            for (int item = pair; item < items && ok; item += pairs) {
                const TilePos p = tile_pos<SPLITK>(item, a.n_tiles, m_tiles, n_splits);
                const int n0 = (p.n * 2 + (int)rank) * kPm, m0 = p.m * BN + (int)rank * (BN / 2);
                for (int kb = k_lo(p); kb < k_hi(p); ++kb, ++it) {
                    const int s = it % S;
                    if (it >= (uint32_t)S && !mbar_wait(empty_bar(s), ((it / S) - 1) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    const bool weights = !WORDS && (!BOX3 || (kb & 1) == 0);  // work items start at an even k block and have an even number of them
                    const uint32_t full = full_bar(it % F);
                    mbar_expect_tx(full, tx_x + (weights ? tx_w : 0u));
                    tma_load_2d(b_tile(s), &map_x, full, kb * kPk, m0);
                    if constexpr (BITS == 0) tma_load_2d(a_tile(s), &map_w, full, kb * kPk, n0);
                    else if (weights) tma_load_2d(p_tile(s), &map_w, full, BOX3 ? kb * (Cfg::P_ROW / 2) : kb * Cfg::P_ROW, n0);
                }
            }
            // no copy is left in flight, even where a wait has run out
            for (uint32_t i = it > (uint32_t)S ? it - (uint32_t)S : 0u; i < it; ++i) (void)mbar_wait(full_bar(i % F), (i / F) & 1, a.status);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ================= MMA issue (first CTA); hand-over (second CTA, bf16) =================
        if (rank == 0) {
            const uint32_t idesc = BITS == 0 ? umma_idesc_bf16(2 * kPm, BN) : umma_idesc_f16(2 * kPm, BN);
            const uint64_t desc_a0 = umma_desc_sw128(a_tile(0)), desc_b0 = umma_desc_sw128(b_tile(0));
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
            uint32_t it = 0, tile_it = 0;
            bool ok = true;
            for (int item = pair; item < items && ok; item += pairs, ++tile_it) {
                const TilePos p = tile_pos<SPLITK>(item, a.n_tiles, m_tiles, n_splits);
                const int buf = tile_it & 1;
                if (tile_it >= 2 && !mbar_wait(tempty_bar(buf), ((tile_it >> 1) - 1) & 1, a.status)) break;
                tcgen05_fence_after();
                const uint32_t d_tmem = tmem_u + (uint32_t)(buf * kMaxRows);
                const int kb_lo = k_lo(p), kb_hi = k_hi(p);
                for (int kb = kb_lo; kb < kb_hi; ++kb, ++it) {
                    const int s = it % S;
                    const uint32_t par = (it / S) & 1;
                    if (BITS == 0 && !mbar_wait(full_bar(s), par, a.status)) ok = false;
                    if (!ok || !mbar_wait(ready_bar(s), par, a.status)) {
                        ok = false;
                        break;
                    }
                    tcgen05_fence_after();
                    const uint64_t stage_off = (uint64_t)(((uint32_t)s * (uint32_t)Cfg::STAGE) >> 4);
                    const uint64_t desc_a = desc_a0 + stage_off, desc_b = desc_b0 + stage_off;
                    if (lane == 0) {
#pragma unroll
                        for (int j = 0; j < kPk / 16; ++j)
                            umma2_ss(d_tmem, desc_a + (uint64_t)(2 * j), desc_b + (uint64_t)(2 * j), idesc, (kb == kb_lo && j == 0) ? 0u : 1u);
                        umma2_commit_both(empty_bar(s));
                    }
                    __syncwarp();
                }
                if (ok && lane == 0) umma2_commit_both(tfull_bar(buf));
                __syncwarp();
            }
            if (it > 0) (void)mbar_wait(empty_bar((it - 1) % S), ((it - 1) / S) & 1, a.status);  // no MMA is left in flight
        } else if (BITS == 0 && lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            const uint32_t to = cluster_map(ready_bar(0), 0);
            for (int item = pair; item < items && ok; item += pairs) {
                const TilePos p = tile_pos<SPLITK>(item, a.n_tiles, m_tiles, n_splits);
                for (int kb = k_lo(p); kb < k_hi(p); ++kb, ++it) {
                    const int s = it % S;
                    if (!mbar_wait(full_bar(s), (it / S) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_pair(to + 8u * s);
                }
            }
        }
        __syncwarp();
    } else if (warp < 2 + Cfg::UW) {
        if constexpr (BITS != 0) {
            // ================= unpack warps: codes -> fp16 weights =================
            const int r = ((warp - 2) & 3) * 32 + lane;  // feature row of this CTA's half of the tile
            constexpr int NG = Cfg::UW / 4;
            const int grp_id = (warp - 2) >> 2;
            const int G = a.K / a.g_size, kb_per_group = a.g_size / kPk;
            const uint32_t to = cluster_map(ready_bar(0), 0);
            uint32_t it0 = 0;
            bool ok = true;
            for (int item = pair; item < items && ok; item += pairs) {
                const TilePos p = tile_pos<SPLITK>(item, a.n_tiles, m_tiles, n_splits);
                const int kb_lo = k_lo(p), kb_hi = k_hi(p);
                const int n = min((p.n * 2 + (int)rank) * kPm + r, a.N - 1);
                UnpackRow<BITS> row;
                row.begin(a.scales + (size_t)n * G, a.zeros + (size_t)n * G, G, WORDS ? a.words + (size_t)n * (a.K / 32 * 3) : nullptr);
                // a group's k blocks: every NG-th, or (3 bits) both of every NG-th pair
                constexpr int RUN = BOX3 ? 2 : 1;
                int kb = kb_lo + RUN * (int)(((uint32_t)grp_id + (uint32_t)NG - it0 / RUN % (uint32_t)NG) % (uint32_t)NG);
                auto next_kb = [&](int k) { return RUN == 1 || (k & 1) ? k + RUN * (NG - 1) + 1 : k + 1; };
                uint32_t w3[12];  // 3-bit codes: a pair's words, in registers when its first k block is handed on
                if (kb < kb_hi) row.fetch(kb, kb / kb_per_group);
                for (int next; kb < kb_hi; kb = next) {
                    const uint32_t it = it0 + (uint32_t)(kb - kb_lo);
                    const int s = it % S;
                    next = next_kb(kb);
                    row.take();
                    if (next < kb_hi) row.fetch(next, next / kb_per_group);
                    if (!mbar_wait(full_bar(it % F), (it / F) & 1, a.status)) {
                        ok = false;
                        break;
                    }
                    const uint32_t src = p_tile(s) + r * Cfg::P_ROW;
                    if constexpr (BOX3) {
                        if ((kb & 1) == 0) {
#pragma unroll
                            for (int i = 0; i < 3; ++i)
                                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                                             : "=r"(w3[4 * i]), "=r"(w3[4 * i + 1]), "=r"(w3[4 * i + 2]), "=r"(w3[4 * i + 3])
                                             : "r"(src + 16 * i));
                            row.set_words(w3[0], w3[1], w3[2], w3[3], w3[4], w3[5]);
                        } else {
                            row.set_words(w3[6], w3[7], w3[8], w3[9], w3[10], w3[11]);
                        }
                    }
                    row.unpack(src, a_tile(s) + r * 128, r);
                    fence_proxy_async_smem();  // the tile must be visible to the tensor core's reads
                    __syncwarp();
                    if (lane == 0) mbar_arrive_pair(to + 8u * s);
                }
                it0 += (uint32_t)(kb_hi - kb_lo);
            }
            __syncwarp();
        }
    } else {
        // ================= epilogue warps =================
        const int q = warp & 3;
        const int c_begin = ((warp - 2 - Cfg::UW) >> 2) * 32;
        const int r = q * 32 + lane;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const int G = BITS == 0 ? 1 : a.K / a.g_size;
        const uint32_t to = cluster_map(tempty_bar(0), 0);
        uint32_t tile_it = 0;
        for (int item = pair; item < items; item += pairs, ++tile_it) {
            const int buf = tile_it & 1;
            const TilePos p = tile_pos<SPLITK>(item, a.n_tiles, m_tiles, n_splits);
            const int n = (p.n * 2 + (int)rank) * kPm + r, m0 = p.m * BN, m_end = min(rows, m0 + BN);
            float fscale = 1.f;
            if constexpr (BITS != 0) fscale = feature_scale(a.scales + (size_t)min(n, a.N - 1) * G, G);
            if (!mbar_wait(tfull_bar(buf), (tile_it >> 1) & 1, a.status)) break;
            tcgen05_fence_after();
#pragma unroll 1
            for (int c0 = c_begin; c0 < BN; c0 += 64) {
                uint32_t u[32];
                tmem_ld_x16(lane_addr + (uint32_t)(buf * kMaxRows + c0), *reinterpret_cast<uint32_t(*)[16]>(&u[0]));
                tmem_ld_x16(lane_addr + (uint32_t)(buf * kMaxRows + c0 + 16), *reinterpret_cast<uint32_t(*)[16]>(&u[16]));
                tmem_ld_wait();
                float xs[32];
                if constexpr (BITS != 0) {
                    // the block's row scales: eight 16-byte loads from one address for the whole warp (the table is padded)
                    const float4 *xp = reinterpret_cast<const float4 *>(a.xscale + m0 + c0);
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4) {
                        const float4 t = m0 + c0 + 4 * q4 < m_end ? __ldg(xp + q4) : make_float4(0.f, 0.f, 0.f, 0.f);
                        xs[4 * q4] = t.x;
                        xs[4 * q4 + 1] = t.y;
                        xs[4 * q4 + 2] = t.z;
                        xs[4 * q4 + 3] = t.w;
                    }
                }
                const bool listed = !SPLITK && a.idx != nullptr;
                const int m_lane = m0 + c0 + lane;
                const int row_lane = (listed && m_lane < m_end) ? a.idx[m_lane] : m_lane;
#pragma unroll
                for (int c = 0; c < 32; ++c) {
                    const int m = m0 + c0 + c;
                    const int row = listed ? __shfl_sync(0xffffffffu, row_lane, c) : m;
                    if (n < a.N && m < m_end) {
                        float v = __uint_as_float(u[c]);
                        if constexpr (BITS != 0) v = (v * xs[c]) * fscale;
                        if constexpr (SPLITK) {
                            a.partial[((size_t)p.split * a.M + m) * a.N + n] = v;
                        } else {
                            if (OUT_F32) reinterpret_cast<float *>(a.Y)[(size_t)row * a.N + n] = v;
                            else reinterpret_cast<__nv_bfloat16 *>(a.Y)[(size_t)row * a.N + n] = __float2bfloat16_rn(v);
                        }
                    }
                }
            }
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_pair(to + 8u * buf);
        }
        __syncwarp();
    }

    // ---- teardown: every role's loop is bounded; nothing is sent to a CTA that has left ----
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tcgen05_fence_after();
        tmem_dealloc2(tmem_base, 512);
    }
}

template <int BITS, bool WORDS, bool OUT_F32, bool SPLITK>
dmr_status_t launch_pair_t(const CUtensorMap &map_w, const CUtensorMap &map_x, const PairArgs &a, int ctas, cudaStream_t st) {
    using Cfg = PairCfg<BITS, WORDS>;
    auto kernel = pair_kernel<BITS, WORDS, OUT_F32, SPLITK>;
    if (!ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), Cfg::SMEM)) return DMR_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3(Cfg::THREADS, 1, 1);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = tc_pdl_enabled() ? 2u : 1u;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, map_w, map_x, a);
    if (e != cudaSuccess) return launch_failed(e);
    return check_launch();
}

template <int BITS, bool WORDS = false>
dmr_status_t launch_pair_bits(const CUtensorMap &map_w, const CUtensorMap &map_x, const PairArgs &a, int ctas, dmr_out_t out, cudaStream_t st) {
    if (a.splits > 1) return launch_pair_t<BITS, WORDS, true, true>(map_w, map_x, a, ctas, st);
    if (out == DMR_OUT_F32) return launch_pair_t<BITS, WORDS, true, false>(map_w, map_x, a, ctas, st);
    return launch_pair_t<BITS, WORDS, false, false>(map_w, map_x, a, ctas, st);
}

}  // namespace

bool pair_supported(int M, int N, int K, int bits, int g) {
    (void)N;
    if (M <= 32 || K % kPk != 0) return false;
    return bits == 0 || ((bits == 3 || bits == 4 || bits == 8) && g % kPk == 0 && K <= kPairMaxK);
}

PairPlan pair_plan(int M, int N, int K, int bits) {
    PairPlan p = {};
    const int pairs = device_sm_count() / 2, nkb = K / kPk;
    p.n_tiles = (N + 2 * kPm - 1) / (2 * kPm);
    // Cycles of a k block at `rows` rows per tile: the MMAs, an SM's intake from the L2, and a floor - the hand-overs, and for codes
    // the unpack warps - below which a k block does not get whatever the tile; plus what a tile costs besides, and, split along k, the partial
    // sums' way to memory and back.  (Measured on the 7B linears, us: floor 330 / 430 / 512 for 4-bit codes: M = 2048 862 / 775 / 750,
    // M = 1000 438 / 394 / 390, M = 4096 1495 / 1442 / 1445; bf16, floor 0 / 400 / 512: M = 700 279 / 269 / 279, M = 1000 355 / 344 / 347.)
    const double a_bytes = bits == 0 ? kPm * kPk * 2 : kPm * kPk * bits / 8;
    const double floor_cycles = bits == 0 ? 400.0 : 512.0;
    double best = -1.0;
    const int most = (M + kMaxRows - 1) / kMaxRows;
    for (int mt = most; mt <= 2 * most + 1; ++mt) {
        const int rows = ((M + mt - 1) / mt + 15) / 16 * 16;
        if (rows < 16) break;
        const int tiles = p.n_tiles * ((M + rows - 1) / rows);
        const double kb_cycles = fmax(fmax(2.0 * rows, (a_bytes + rows * kPk) / 61.0), floor_cycles);
        for (int sp = 1; sp <= 8; ++sp) {
            if (sp > 1 && (tiles >= pairs || nkb / sp < 16)) break;
            int per = (nkb + sp - 1) / sp;
            if (bits == 3 && nkb % 2 == 0) per = (per + 1) / 2 * 2;  // two k blocks share a box
            const int splits = (nkb + per - 1) / per;
            const int rounds = (tiles * splits + pairs - 1) / pairs;
            double cost = rounds * (per * kb_cycles + 1500.0);
            if (splits > 1) cost += 6000.0 + (2.0 * splits) * M * (double)N * 4.0 / 3000.0;
            if (best < 0.0 || cost < best) {
                best = cost;
                p.rows = rows;
                p.splits = splits;
                p.kb_per_split = per;
            }
        }
    }
    p.tiles = p.n_tiles * ((M + p.rows - 1) / p.rows);
    const int items = p.tiles * p.splits;
    p.ctas = 2 * (items < pairs ? items : pairs);
    p.partial_bytes = p.splits > 1 ? (size_t)p.splits * M * N * sizeof(float) : 0;
    return p;
}

dmr_status_t launch_pair(const uint16_t *X, int M, RowSel sel, const float *xscale, const void *weights, const uint16_t *scales,
                         const uint8_t *zeros, int N, int K, int bits, int g, void *Y, dmr_out_t out, float *partial, int32_t *status,
                         cudaStream_t st) {
    const PairPlan p = pair_plan(M, N, K, bits);
    if (p.splits > 1 && !partial) return DMR_ERR_WORKSPACE;
    CUtensorMap map_w, map_x;
    if (!make_tensor_map_2d(&map_x, bits == 0 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, X, (uint64_t)M, (uint64_t)K,
                            (uint64_t)K * 2, (uint32_t)(p.rows / 2), kPk, TmaSwizzle::k128B))
        return DMR_ERR_CUDA;
    const uint64_t row_bytes = (uint64_t)K * bits / 8;
    const bool words = bits == 3 && K % (2 * kPk) != 0;
    if (bits == 0) {
        if (!make_tensor_map_2d(&map_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, weights, (uint64_t)N, (uint64_t)K, (uint64_t)K * 2, kPm, kPk, TmaSwizzle::k128B))
            return DMR_ERR_CUDA;
    } else if (words) {
        map_w = map_x;  // (not used)
    } else if (!make_tensor_map_2d(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, weights, (uint64_t)N, row_bytes, row_bytes, kPm,
                                   (uint32_t)(bits == 3 ? 48 : kPk * bits / 8), TmaSwizzle::kNone)) {
        return DMR_ERR_CUDA;
    }
    PairArgs a = {};
    a.scales = scales;
    a.zeros = zeros;
    a.words = words ? reinterpret_cast<const uint32_t *>(weights) : nullptr;
    a.xscale = xscale;
    a.Y = Y;
    a.idx = sel.idx;
    a.count = sel.count;
    a.status = status;
    a.partial = p.splits > 1 ? partial : nullptr;
    a.M = M;
    a.N = N;
    a.K = K;
    a.g_size = bits == 0 ? K : g;
    a.n_tiles = p.n_tiles;
    a.tile_rows = p.rows;
    a.splits = p.splits;
    a.kb_per_split = p.kb_per_split;
    dmr_status_t r;
    if (bits == 0) r = launch_pair_bits<0>(map_w, map_x, a, p.ctas, out, st);
    else if (words) r = launch_pair_bits<3, true>(map_w, map_x, a, p.ctas, out, st);
    else if (bits == 3) r = launch_pair_bits<3>(map_w, map_x, a, p.ctas, out, st);
    else if (bits == 4) r = launch_pair_bits<4>(map_w, map_x, a, p.ctas, out, st);
    else r = launch_pair_bits<8>(map_w, map_x, a, p.ctas, out, st);
    if (r != DMR_OK || p.splits == 1) return r;
    return launch_splitk_reduce(partial, p.splits, M, N, sel, Y, out, st);
}

}  // namespace dmr
