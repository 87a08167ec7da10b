// The router's forward pass (see router_fwd.cu for the method) as ONE cooperative launch of thread-block clusters, for calls of up
// to some hundreds of tokens (fused_cost says how many): an agent, or some tens of them, asking for the precision of their next step.
//
// What bounds it.  One step of one agent (32 tokens, d = 384, 8 layers) reads 57 MB of parameters for 0.9 GFLOP: 9 us of HBM time.
// As 58 dependent kernels it took 475 us on the device (580 with their launches): each paid a launch, a cold start and the latency of
// its first loads.  Here the layers run inside one kernel, and the steps between them cost a barrier of a cluster (hardware, below a
// microsecond) instead of a launch.  Measured, calls one after the other with parameters that have left the L2: one step 582 -> 220 us, 8 steps
// of up to 32 entries 1641 -> 369, 20 steps 1763 -> 752, 40 steps 2110 -> 1373.  What is left of a layer's 26 us at one step is latency: the grid
// barrier 4.7, attention 2.9, the linears 8 (weights of a warp's second task are not hidden), the exchanges and layer norms 10.  (768 threads
// with 80 registers spilled the weights held across the barriers: 318 us; six features per lane, so that one task per warp is enough: 232.)
//
// Split.  The valid tokens (padded ones are dropped) are dealt out evenly to clusters of 16 CTAs; every CTA of a cluster holds a
// copy of its tokens' activations in shared memory and computes a sixteenth of the output features of every linear, so an SM
// reads a sixteenth of the parameters (3.5 MB in all, about 30 us at an SM's intake from the L2) and the clusters share them in the L2,
// into which a layer's parameters are requested a layer ahead.
// Outputs go to the other CTAs through distributed shared memory.  The feed-forward block keeps its hidden features where they
// are computed (the second linear is split along k) and exchanges partial sums instead: a quarter of the traffic.  Only
// keys and values cross clusters, through global memory and one grid-wide barrier per layer (two buffers, so that a fast
// cluster never overwrites what a slow one still reads).  In the last layer only the last valid step of a sequence is
// carried past the keys and values, and those steps are dealt out to the clusters again.
//
// Linears.  A warp takes tasks of 16 features x 96 inputs: lane (r, k) (r = lane / 8, k = lane % 8) holds four features' weights for three
// groups of four inputs in registers - requested before the barrier that ends the step before, so their latency is hidden -
// and meets them with four tokens at a time; eight lanes' sums are added by shuffles, the k ranges' sums in order through shared
// memory.  fp32 fused multiply-adds throughout, every sum in a fixed order that depends on the layer's sizes only.
#include "sm100.cuh"

namespace dmr {

namespace {

constexpr int kCs = 16;                   // CTAs per cluster
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kRows = 4;                  // features a lane holds the weights of
constexpr int kTaskRows = 4 * kRows, kTaskK = 96;
constexpr int kTokBlock = 32;             // tokens a cluster works on at a time
constexpr int kAttWarps = 4;              // warps that share the keys of a (token, head)
constexpr float kEps = 1e-5f;

struct FusedArgs {
    const float *params, *Z;
    const int32_t *lengths;
    float *probs, *scores;
    float *H;              // [T][d] a layer's input, compact token rows
    float *QKV;            // two buffers [T][3 d]
    uint32_t *counter;     // grid barrier, then whether this launch takes the call; zero at launch
    long long limit;       // work (see router_work) up to which it does
    int B, L, d, heads, dh, ffn, layers, l_max, classes, score_class;
    int rq, rd, rf;        // features per CTA of QKV, of the d-wide linears, of the hidden layer (multiples of 4)
    int off_ss, off_as, off_fs, off_par, off_part, off_tab;  // shared memory, in floats
};

// Tokens times layers: past the keys and values of the last layer there is one token per sequence.
__host__ __device__ constexpr long long router_work(int layers, long long tokens, int B) { return (layers - 1) * tokens + B; }

__device__ __forceinline__ int seq_len(int n, int L) { return n < 1 ? 1 : (n > L ? L : n); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_f4(uint32_t addr, const float4 &v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// A load that stays where it is written (the compiler would move it behind the barrier that is to hide it).
__device__ __forceinline__ float4 ldg_early(const float *p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 add4(const float4 &a, const float4 &b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

struct Weights {
    float4 w[kRows][3];
};

// A linear's share of this CTA: features [0, rows) of `W` (already advanced to the CTA's first), inputs [0, K).
struct Linear {
    const float *W;
    int ld, rows, K, ks;  // ks = ceil(K / kTaskK)
    __device__ __forceinline__ int tasks() const { return (rows + kTaskRows - 1) / kTaskRows * ks; }
};

__device__ __forceinline__ void load_task(Weights &t, const Linear &l, int task, int lane) {
    const int rl = lane >> 3, kl = lane & 7;
    const int row = task / l.ks * kTaskRows + rl * kRows, k = task % l.ks * kTaskK + kl * 4;
    const float *p = l.W + (size_t)row * l.ld + k;
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
        for (int i = 0; i < 3; ++i)
            t.w[r][i] = row + r < l.rows && k + 32 * i < l.K ? ldg_early(p + (size_t)r * l.ld + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// part[task][token][16 features] = this task's sums for tokens [0, tc) of x (rows of `xs` floats).
__device__ __forceinline__ void run_task(const Weights &t, const Linear &l, int task, int lane, const float *x, int xs, int tc, float *part) {
    const int rl = lane >> 3, kl = lane & 7;
    const int k = task % l.ks * kTaskK + kl * 4;
    const float *x0 = x + (k < l.K ? k : 0);
    const int o1 = k + 32 < l.K ? 32 : 0, o2 = k + 64 < l.K ? 64 : 0;  // past the end: weights are zero, any finite x does
    const bool b2 = kl & 4, b1 = kl & 2, b0 = kl & 1;
    float *out = part + (size_t)task * kTokBlock * kTaskRows + ((b2 ? 2 : 0) + (b1 ? 1 : 0)) * kTaskRows + rl * kRows + (b0 ? kRows / 2 : 0);
#pragma unroll 1
    for (int tb = 0; tb < tc; tb += 4) {
        float acc[4][kRows];  // [token][feature]
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 a = *reinterpret_cast<const float4 *>(x0 + u * xs);
#pragma unroll
            for (int r = 0; r < kRows; ++r) acc[u][r] = fmaf(t.w[r][0].w, a.w, fmaf(t.w[r][0].z, a.z, fmaf(t.w[r][0].y, a.y, t.w[r][0].x * a.x)));
            const float4 b = *reinterpret_cast<const float4 *>(x0 + u * xs + o1);
#pragma unroll
            for (int r = 0; r < kRows; ++r) acc[u][r] = fmaf(t.w[r][1].w, b.w, fmaf(t.w[r][1].z, b.z, fmaf(t.w[r][1].y, b.y, fmaf(t.w[r][1].x, b.x, acc[u][r]))));
            const float4 c = *reinterpret_cast<const float4 *>(x0 + u * xs + o2);
#pragma unroll
            for (int r = 0; r < kRows; ++r) acc[u][r] = fmaf(t.w[r][2].w, c.w, fmaf(t.w[r][2].z, c.z, fmaf(t.w[r][2].y, c.y, fmaf(t.w[r][2].x, c.x, acc[u][r]))));
        }
        x0 += 4 * xs;
        // eight lanes' sums: every step keeps half of the values, so lane k ends with token k / 2's features 2 (k % 2), + 1
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const float send = b2 ? acc[u][r] : acc[2 + u][r], keep = b2 ? acc[2 + u][r] : acc[u][r];
                acc[u][r] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 4);
            }
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const float send = b1 ? acc[0][r] : acc[1][r], keep = b1 ? acc[1][r] : acc[0][r];
            acc[0][r] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 2);
        }
#pragma unroll
        for (int r = 0; r < kRows / 2; ++r) {
            const float send = b0 ? acc[0][r] : acc[0][kRows / 2 + r], keep = b0 ? acc[0][kRows / 2 + r] : acc[0][r];
            out[r] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 1);
        }
        out += 4 * kTaskRows;
    }
}

// All tasks of a linear; the warp's first one is in `t` already.
__device__ __forceinline__ void run_linear(Weights &t, const Linear &l, const float *x, int xs, int tc, float *part) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 1
    for (int task = warp; task < l.tasks(); task += kWarps) {
        if (task != warp) load_task(t, l, task, lane);
        run_task(t, l, task, lane, x, xs, tc, part);
    }
    __syncthreads();
}
__device__ __forceinline__ void prefetch_linear(Weights &t, const Linear &l) {
    const int warp = threadIdx.x >> 5;
    if (warp < l.tasks()) load_task(t, l, warp, threadIdx.x & 31);
}
// Features 4 q .. 4 q + 3 of token i, the k ranges added in order.
__device__ __forceinline__ float4 sum_quad(const Linear &l, const float *part, int q, int i) {
    const int row = 4 * q;
    const float *p = part + ((size_t)(row / kTaskRows * l.ks) * kTokBlock + i) * kTaskRows + row % kTaskRows;
    float4 v = *reinterpret_cast<const float4 *>(p);
    for (int s = 1; s < l.ks; ++s) v = add4(v, *reinterpret_cast<const float4 *>(p + (size_t)s * kTokBlock * kTaskRows));
    return v;
}

// x[i][:] = LN(s[i][:]) g + b for tokens [0, tc), a warp per token.
__device__ __forceinline__ void layer_norm(const float *s, const float *g, const float *b, int d, int tc, float *x) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < tc; i += kWarps) {
        const float *row = s + (size_t)i * d;
        float sum = 0.f;
        for (int c = lane * 4; c < d; c += 128) {
            const float4 v = *reinterpret_cast<const float4 *>(row + c);
            sum += (v.x + v.y) + (v.z + v.w);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        const float mean = sum / (float)d;
        float sq = 0.f;
        for (int c = lane * 4; c < d; c += 128) {
            const float4 v = *reinterpret_cast<const float4 *>(row + c);
            const float e0 = v.x - mean, e1 = v.y - mean, e2 = v.z - mean, e3 = v.w - mean;
            sq = fmaf(e0, e0, fmaf(e1, e1, fmaf(e2, e2, fmaf(e3, e3, sq))));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
        const float rstd = 1.f / sqrtf(sq / (float)d + kEps);
        for (int c = lane * 4; c < d; c += 128) {
            const float4 v = *reinterpret_cast<const float4 *>(row + c);
            const float4 gg = *reinterpret_cast<const float4 *>(g + c), bb = *reinterpret_cast<const float4 *>(b + c);
            *reinterpret_cast<float4 *>(x + (size_t)i * d + c) =
                make_float4((v.x - mean) * rstd * gg.x + bb.x, (v.y - mean) * rstd * gg.y + bb.y, (v.z - mean) * rstd * gg.z + bb.z, (v.w - mean) * rstd * gg.w + bb.w);
        }
    }
    __syncthreads();
}

// Attention of a token and head over the keys j0, j0 + 4, ... (n in all) by one of the four warps that share it: a key is met by
// DH / 4 lanes with four columns each, eight keys' rows of K and V are requested before the first is used.  out[0 .. DH) = the weighted
// sum of the values, out[DH] = the largest score, out[DH + 1] = the sum of the weights.
template <int DH>
__device__ __forceinline__ void attend(const float *q, const float *kbase, const float *vbase, int ld, int j0, int n, float *out) {
    constexpr int F4 = DH / 4, GROUPS = 32 / F4, U = 8 / GROUPS > 0 ? 8 / GROUPS : 1;  // U keys per lane at a time
    const int lane = threadIdx.x & 31, grp = lane / F4, col = lane % F4;
    const float4 qv = __ldcg(reinterpret_cast<const float4 *>(q) + col);
    const float scale = 1.0f / sqrtf((float)DH);
    float mx = -INFINITY, sum = 0.f;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j = j0; j < n; j += kAttWarps * U * GROUPS) {
        float4 kv[U], vv[U];
        float s[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const size_t row = (size_t)min(j + kAttWarps * (u * GROUPS + grp), n - 1) * ld;
            kv[u] = __ldcg(reinterpret_cast<const float4 *>(kbase + row) + col);
            vv[u] = __ldcg(reinterpret_cast<const float4 *>(vbase + row) + col);
        }
        float top = mx;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float v = qv.x * kv[u].x;
            v = fmaf(qv.y, kv[u].y, v);
            v = fmaf(qv.z, kv[u].z, v);
            v = fmaf(qv.w, kv[u].w, v);
#pragma unroll
            for (int x = 1; x < F4; x <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, x);
            s[u] = j + kAttWarps * (u * GROUPS + grp) < n ? v * scale : -INFINITY;
            top = fmaxf(top, s[u]);
        }
#pragma unroll
        for (int x = F4; x < 32; x <<= 1) top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, x));
        const float r = expf(mx - top);  // 0 the first time
        mx = top;
        sum *= r;
        o.x *= r;
        o.y *= r;
        o.z *= r;
        o.w *= r;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float e = expf(s[u] - top);
            sum += e;
            o.x = fmaf(e, vv[u].x, o.x);
            o.y = fmaf(e, vv[u].y, o.y);
            o.z = fmaf(e, vv[u].z, o.z);
            o.w = fmaf(e, vv[u].w, o.w);
        }
    }
#pragma unroll
    for (int x = F4; x < 32; x <<= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, x);
        o.x += __shfl_xor_sync(0xFFFFFFFFu, o.x, x);
        o.y += __shfl_xor_sync(0xFFFFFFFFu, o.y, x);
        o.z += __shfl_xor_sync(0xFFFFFFFFu, o.z, x);
        o.w += __shfl_xor_sync(0xFFFFFFFFu, o.w, x);
    }
    if (grp == 0) *reinterpret_cast<float4 *>(out + 4 * col) = o;
    if (lane == 0) {
        out[DH] = mx;
        out[DH + 1] = sum;
    }
}

// Requests floats [0, n) of p into the L2, this CTA's share of them (by one thread).
__device__ __forceinline__ void prefetch_l2(const float *p, size_t n) {
    const size_t per = (n / 4 + gridDim.x - 1) / gridDim.x * 4, lo = per * blockIdx.x;  // multiples of 16 bytes
    if (lo >= n) return;
    const uint32_t bytes = (uint32_t)((n - lo < per ? n - lo : per) * sizeof(float)) & ~15u;
    if (bytes) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p + lo), "r"(bytes) : "memory");
}

// All CTAs of the grid (they are co-resident: cooperative launch).  `target` = CTAs x number of this barrier.
__device__ __forceinline__ bool grid_barrier(uint32_t *counter, uint32_t target) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
        uint32_t seen = 0;
        ok = false;
        for (uint32_t i = 0; i < kWaitLimit; ++i) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
            if (seen >= target) {
                ok = true;
                break;
            }
        }
    }
    return __syncthreads_or(threadIdx.x == 0 && !ok) == 0;
}

template <int DH>
__global__ void __launch_bounds__(kThreads, 1) router_fused_kernel(const FusedArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_ctarank(), cid = (int)cluster_id_x(), clusters = (int)cluster_count_x();
    const int d = a.d, f = a.ffn;
    float *xs = sm;                   // [tokens][d]  the layer's input (replicated in the cluster, like the next two)
    float *ss = sm + a.off_ss;        // [tokens][d]  sums before a layer norm
    float *as = sm + a.off_as;        // [tokens][d]  attention output; later the partial sums sent here, [16 senders][tokens][rd]
    float *fs = sm + a.off_fs;        // [tokens][rf] this CTA's hidden features
    // the layer's vectors: ln1_g, ln1_b, ln2_g, ln2_b [d], then this CTA's share of bo, b2 [rd], b1 [rf] and the next layer's bqkv [rq]
    float *par = sm + a.off_par;
    float *part = sm + a.off_part;    // [tasks][tokens][16]
    int *start = reinterpret_cast<int *>(sm + a.off_tab);  // [B + 1] first compact row of each sequence
    int *tseq = start + a.B + 1;      // [tokens] the block's tokens: sequence, and step
    int *tstep = tseq + kTokBlock;
    const size_t layer_floats = (size_t)4 * d * d + (size_t)2 * f * d + 9 * (size_t)d + f;

    if (threadIdx.x == 0) prefetch_l2(a.params + (size_t)a.l_max * d, layer_floats);
    // A CTA without hidden features (sixteen shares of a multiple of four can be more than there are) runs the second linear's tasks with weights
    // of zero and reads four floats of each of these rows for them: what an earlier kernel left there may not be finite.
    if (threadIdx.x < kTokBlock) *reinterpret_cast<float4 *>(fs + threadIdx.x * a.rf) = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp == 0) {  // first rows: a running sum of the lengths
        int base = 0;
        for (int b0 = 0; b0 < a.B; b0 += 32) {
            const int n = b0 + lane < a.B ? seq_len(a.lengths[b0 + lane], a.L) : 0;
            int v = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xFFFFFFFFu, v, o);
                if (lane >= o) v += u;
            }
            if (b0 + lane < a.B) start[b0 + lane] = base + v - n;
            base += __shfl_sync(0xFFFFFFFFu, v, 31);
        }
        if (lane == 0) start[a.B] = base;
    }
    __syncthreads();
    const int total = start[a.B];
    if (router_work(a.layers, total, a.B) > a.limit) return;  // every CTA finds the same
    if (blockIdx.x == 0 && threadIdx.x == 0) a.counter[1] = 1u;
    const int row_lo = (int)((long long)total * cid / clusters), row_hi = (int)((long long)total * (cid + 1) / clusters);
    const int seq_lo = (int)((long long)a.B * cid / clusters), seq_hi = (int)((long long)a.B * (cid + 1) / clusters);
    const size_t buf = (size_t)a.B * a.L * 3 * d;

    const int q0 = rank * a.rq, d0 = rank * a.rd, f0 = rank * a.rf;
    const int qn = max(0, min(a.rq, 3 * d - q0)), dn = max(0, min(a.rd, d - d0)), fn = max(0, min(a.rf, f - f0));
    const int kd = (d + kTaskK - 1) / kTaskK, kf = (a.rf + kTaskK - 1) / kTaskK;

    float *s_ln1g = par, *s_ln1b = s_ln1g + d, *s_ln2g = s_ln1b + d, *s_ln2b = s_ln2g + d;
    float *s_bo = s_ln2b + d, *s_b2 = s_bo + a.rd, *s_b1 = s_b2 + a.rd, *s_bqkv = s_b1 + a.rf;

    Weights w;
    uint32_t barriers = 0;
    bool ok = true;

    // The tokens of a block: rows lo + [0, tc), or in the last layer the last steps of sequences lo + [0, tc).
    auto set_tokens = [&](int lo, int tc, bool last) {
        __syncthreads();  // the block before is done with the tables
        if ((int)threadIdx.x < tc) {
            int b = lo + (int)threadIdx.x, step;
            if (last) {
                step = start[b + 1] - start[b] - 1;
            } else {
                const int row = b;
                int x = 0, y = a.B;  // start[x] <= row < start[y]
                while (y - x > 1) {
                    const int m = (x + y) / 2;
                    if (start[m] <= row) x = m;
                    else y = m;
                }
                b = x;
                step = row - start[x];
            }
            tseq[threadIdx.x] = b;
            tstep[threadIdx.x] = step;
        }
        __syncthreads();
    };
    // x of the block's tokens, from the embeddings (first) or from H
    auto load_x = [&](int tc, bool first) {
        const int d4 = d / 4;
        for (int e = threadIdx.x; e < tc * d4; e += kThreads) {
            const int i = e / d4, c = e % d4;
            float4 v;
            if (first) {
                v = add4(__ldg(reinterpret_cast<const float4 *>(a.Z + ((size_t)tseq[i] * a.L + tstep[i]) * d) + c),
                         __ldg(reinterpret_cast<const float4 *>(a.params + (size_t)tstep[i] * d) + c));
            } else {
                v = __ldcg(reinterpret_cast<const float4 *>(a.H + (size_t)(start[tseq[i]] + tstep[i]) * d) + c);
            }
            *reinterpret_cast<float4 *>(xs + (size_t)i * d + 4 * c) = v;
        }
        __syncthreads();
    };
    auto store_h = [&](int tc) {
        for (int i = rank + kCs * warp; i < tc; i += kCs * kWarps)
            for (int c = lane * 4; c < d; c += 128)
                *reinterpret_cast<float4 *>(a.H + (size_t)(start[tseq[i]] + tstep[i]) * d + c) = *reinterpret_cast<const float4 *>(xs + (size_t)i * d + c);
    };
    auto qkv_linear = [&](int layer) -> Linear {
        return {a.params + (size_t)a.l_max * d + (size_t)layer * layer_floats + (size_t)q0 * d, d, qn, d, kd};
    };
    // Q, K, V of `layer` for the block in xs, to global memory; the weights of the warp's first task are in w.
    auto project = [&](int layer, int tc) {
        const Linear l = qkv_linear(layer);
        run_linear(w, l, xs, d, tc, part);
        const float *bias = s_bqkv;
        float *out = a.QKV + (layer & 1) * buf;
        for (int e = threadIdx.x; e < qn / 4 * tc; e += kThreads) {
            const int q = e % (qn / 4), i = e / (qn / 4);
            const float4 v = add4(sum_quad(l, part, q, i), *reinterpret_cast<const float4 *>(bias + 4 * q));
            *reinterpret_cast<float4 *>(out + (size_t)(start[tseq[i]] + tstep[i]) * (3 * d) + q0 + 4 * q) = v;
        }
    };
    // This CTA's features d0 .. of ss to the other CTAs, a warp for each of them.
    static_assert(kWarps == kCs, "one warp per CTA of the cluster");
    auto broadcast_ss = [&](int tc) {
        __syncthreads();
        const int nq = dn / 4;
        if (warp != rank) {
            const uint32_t to = cluster_map(smem_u32(ss + d0), (uint32_t)warp);
            for (int e = lane; e < nq * tc; e += 32) {
                const int i = e / nq, at = i * d + 4 * (e - i * nq);
                st_cluster_f4(to + 4u * (uint32_t)at, *reinterpret_cast<const float4 *>(ss + d0 + at));
            }
        }
        __syncwarp();
    };
    // Starts copying n floats (a multiple of 4) to shared memory.
    auto copy_async = [&](float *dst, const float *src, int n) {
        for (int e = threadIdx.x; e < n / 4; e += kThreads)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + 4 * e)), "l"(src + 4 * e) : "memory");
    };
    auto bqkv = [&](int layer) { return a.params + (size_t)a.l_max * d + (size_t)layer * layer_floats + (size_t)3 * d * d + q0; };

    copy_async(s_bqkv, bqkv(0), qn);
    asm volatile("cp.async.wait_all;" ::: "memory");  // seen by the others behind the next __syncthreads

    for (int lo = row_lo; lo < row_hi; lo += kTokBlock) {
        const int tc = min(kTokBlock, row_hi - lo);
        prefetch_linear(w, qkv_linear(0));
        set_tokens(lo, tc, false);
        load_x(tc, true);
        store_h(tc);
        project(0, tc);
    }
    const bool one_block = row_hi - row_lo <= kTokBlock;

    for (int layer = 0; layer < a.layers; ++layer) {
        const bool last = layer == a.layers - 1;
        const float *p = a.params + (size_t)a.l_max * d + (size_t)layer * layer_floats;
        const float *wo = p + (size_t)3 * d * d + 3 * d, *bo = wo + (size_t)d * d, *ln1_g = bo + d, *ln1_b = ln1_g + d, *w1 = ln1_b + d, *b1 = w1 + (size_t)f * d;
        const float *w2 = b1 + f, *b2 = w2 + (size_t)d * f, *ln2_g = b2 + d, *ln2_b = ln2_g + d;
        const Linear lo_l = {wo + (size_t)d0 * d, d, dn, d, kd};
        const Linear l1 = {w1 + (size_t)f0 * d, d, fn, d, kd};
        const Linear l2 = {w2 + f0, f, d, fn, kf};
        ok = grid_barrier(a.counter, ++barriers * gridDim.x) && ok;
        if (threadIdx.x == 0 && !last) prefetch_l2(p + layer_floats, layer_floats);
        copy_async(s_ln1g, ln1_g, 2 * d);  // gain and offset lie side by side
        copy_async(s_ln2g, ln2_g, 2 * d);
        copy_async(s_bo, bo + d0, dn);
        copy_async(s_b2, b2 + d0, dn);
        copy_async(s_b1, b1 + f0, fn);
        if (!last) copy_async(s_bqkv, bqkv(layer + 1), qn);
        const float *qkv = a.QKV + (layer & 1) * buf;
        const int lo_i = last ? seq_lo : row_lo, hi_i = last ? seq_hi : row_hi;
        for (int lo = lo_i; lo < hi_i; lo += kTokBlock) {
            const int tc = min(kTokBlock, hi_i - lo);
            if (last || !one_block) {
                set_tokens(lo, tc, last);
                load_x(tc, false);
            }
            // ---- attention: four warps per (token, head), the pairs spread over the CTAs; partial results meet in `part` ----
            constexpr int AS = DH + 4;  // floats per partial result
            const int pairs = tc * a.heads, mine = pairs > rank ? (pairs - rank + kCs - 1) / kCs : 0;
            for (int e = warp; e < kAttWarps * mine; e += kWarps) {
                const int pr = rank + kCs * (e / kAttWarps), i = pr / a.heads, h = pr % a.heads;
                const int first = start[tseq[i]], n = start[tseq[i] + 1] - first;
                const float *base = qkv + (size_t)first * (3 * d) + h * DH;
                attend<DH>(base + (size_t)tstep[i] * (3 * d), base + d, base + 2 * d, 3 * d, e % kAttWarps, n, part + (size_t)e * AS);
            }
            asm volatile("cp.async.wait_all;" ::: "memory");  // the layer's vectors
            __syncthreads();
            constexpr int F4 = DH / 4;
            for (int e = lane; e < mine * F4; e += 32) {  // every warp for one CTA of the cluster
                const int c = e % F4, to = warp, m = e / F4;
                const int pr = rank + kCs * m, i = pr / a.heads, h = pr % a.heads;
                const float *r = part + (size_t)(kAttWarps * m) * AS;
                float top = r[DH];
#pragma unroll
                for (int s = 1; s < kAttWarps; ++s) top = fmaxf(top, r[s * AS + DH]);
                float sum = 0.f;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int s = 0; s < kAttWarps; ++s) {  // a warp without keys: largest score -inf, weight 0
                    const float g = expf(r[s * AS + DH] - top);
                    const float4 v = *reinterpret_cast<const float4 *>(r + s * AS + 4 * c);
                    sum = fmaf(g, r[s * AS + DH + 1], sum);
                    o.x = fmaf(g, v.x, o.x);
                    o.y = fmaf(g, v.y, o.y);
                    o.z = fmaf(g, v.z, o.z);
                    o.w = fmaf(g, v.w, o.w);
                }
                const float inv = 1.f / sum;
                st_cluster_f4(cluster_map(smem_u32(as + (size_t)i * d + h * DH + 4 * c), (uint32_t)to), make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv));
            }
            __syncwarp();
            cluster_arrive();
            prefetch_linear(w, lo_l);
            cluster_wait();
            // ---- output projection, residual ----
            run_linear(w, lo_l, as, d, tc, part);
            for (int e = threadIdx.x; e < dn / 4 * tc; e += kThreads) {
                const int q = e % (dn / 4), i = e / (dn / 4);
                const float4 v = add4(add4(sum_quad(lo_l, part, q, i), *reinterpret_cast<const float4 *>(s_bo + 4 * q)),
                                      *reinterpret_cast<const float4 *>(xs + (size_t)i * d + d0 + 4 * q));
                *reinterpret_cast<float4 *>(ss + (size_t)i * d + d0 + 4 * q) = v;
            }
            broadcast_ss(tc);
            cluster_arrive();
            prefetch_linear(w, l1);
            cluster_wait();
            layer_norm(ss, s_ln1g, s_ln1b, d, tc, xs);
            // ---- feed-forward: this CTA's hidden features, and what they add to every output ----
            run_linear(w, l1, xs, d, tc, part);
            for (int e = threadIdx.x; e < fn / 4 * tc; e += kThreads) {
                const int q = e % (fn / 4), i = e / (fn / 4);
                const float4 v = add4(sum_quad(l1, part, q, i), *reinterpret_cast<const float4 *>(s_b1 + 4 * q));
                *reinterpret_cast<float4 *>(fs + (size_t)i * a.rf + 4 * q) = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
            }
            prefetch_linear(w, l2);
            __syncthreads();
            run_linear(w, l2, fs, a.rf, tc, part);
            for (int e = threadIdx.x; e < d / 4 * tc; e += kThreads) {
                const int q = e % (d / 4), i = e / (d / 4), to = 4 * q / a.rd;
                const float4 v = sum_quad(l2, part, q, i);
                st_cluster_f4(cluster_map(smem_u32(as + ((size_t)rank * kTokBlock + i) * a.rd + (4 * q - to * a.rd)), (uint32_t)to), v);
            }
            cluster_arrive();
            cluster_wait();
            for (int e = threadIdx.x; e < dn / 4 * tc; e += kThreads) {
                const int q = e % (dn / 4), i = e / (dn / 4);
                float4 v = *reinterpret_cast<const float4 *>(as + (size_t)i * a.rd + 4 * q);
#pragma unroll
                for (int s = 1; s < kCs; ++s) v = add4(v, *reinterpret_cast<const float4 *>(as + ((size_t)s * kTokBlock + i) * a.rd + 4 * q));
                v = add4(add4(v, *reinterpret_cast<const float4 *>(s_b2 + 4 * q)), *reinterpret_cast<const float4 *>(xs + (size_t)i * d + d0 + 4 * q));
                *reinterpret_cast<float4 *>(ss + (size_t)i * d + d0 + 4 * q) = v;
            }
            broadcast_ss(tc);
            cluster_arrive();
            if (!last) prefetch_linear(w, qkv_linear(layer + 1));
            cluster_wait();
            layer_norm(ss, s_ln2g, s_ln2b, d, tc, xs);
            if (!last) {
                if (!one_block || layer == a.layers - 2) store_h(tc);
                project(layer + 1, tc);
                continue;
            }
            // ---- head: a warp per sequence, spread over the CTAs ----
            const float *wc = a.params + (size_t)a.l_max * d + (size_t)a.layers * layer_floats, *bc = wc + (size_t)a.classes * d;
            for (int i = rank + kCs * warp; i < tc; i += kCs * kWarps) {
                const float *hstar = xs + (size_t)i * d;
                float mine_l = -INFINITY;  // lane c keeps the logit of class c
                for (int c = 0; c < a.classes; ++c) {
                    float v = 0.f;
                    for (int k = lane; k < d; k += 32) v = fmaf(__ldg(wc + (size_t)c * d + k), hstar[k], v);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
                    if (lane == c) mine_l = v + __ldg(bc + c);
                }
                float mx = mine_l;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
                const float e = lane < a.classes ? expf(mine_l - mx) : 0.f;
                float sum = e;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
                const float pr = ok ? e / sum : NAN;  // a grid barrier ran out: no answer
                if (lane < a.classes) a.probs[(size_t)tseq[i] * a.classes + lane] = pr;
                if (a.scores && lane == a.score_class) a.scores[tseq[i]] = pr;
            }
        }
    }
}

struct FusedPlan {
    FusedArgs a;
    size_t smem;
};

FusedPlan fused_plan(const dmr_router_cfg_t &c, int B, int L) {
    FusedPlan p = {};
    FusedArgs &a = p.a;
    const auto share = [](int n) { return ((n + kCs - 1) / kCs + 3) / 4 * 4; };
    a.B = B;
    a.L = L;
    a.d = c.d;
    a.heads = c.heads;
    a.dh = c.d / c.heads;
    a.ffn = c.ffn;
    a.layers = c.layers;
    a.l_max = c.l_max;
    a.classes = c.classes;
    a.rq = share(3 * c.d);
    a.rd = share(c.d);
    a.rf = share(c.ffn);
    const auto groups = [](int rows) { return (rows + kTaskRows - 1) / kTaskRows; };
    const int kd = (c.d + kTaskK - 1) / kTaskK, kf = (a.rf + kTaskK - 1) / kTaskK;
    int tasks = groups(a.rq) * kd;
    if (groups(a.rf) * kd > tasks) tasks = groups(a.rf) * kd;
    if (groups(c.d) * kf > tasks) tasks = groups(c.d) * kf;
    size_t off = (size_t)kTokBlock * c.d;
    a.off_ss = (int)off;
    off += (size_t)kTokBlock * c.d;
    a.off_as = (int)off;
    off += (size_t)kTokBlock * kCs * a.rd;
    a.off_fs = (int)off;
    off += (size_t)kTokBlock * a.rf;
    a.off_par = (int)off;
    off += (size_t)4 * c.d + 2 * a.rd + a.rf + a.rq;
    a.off_part = (int)off;
    // the attention's partial results use `part` too: four per (token, head) of this CTA
    const size_t sums = (size_t)tasks * kTokBlock * kTaskRows, att = (size_t)kAttWarps * ((kTokBlock * c.heads + kCs - 1) / kCs) * (a.dh + 4);
    off += sums > att ? sums : att;
    a.off_tab = (int)off;
    off += (size_t)B + 1 + 2 * kTokBlock;
    p.smem = off * sizeof(float);
    return p;
}

using FusedKernel = void (*)(FusedArgs);
FusedKernel fused_kernel(int dh) {
    switch (dh) {
        case 16: return router_fused_kernel<16>;
        case 32: return router_fused_kernel<32>;
        case 64: return router_fused_kernel<64>;
        case 128: return router_fused_kernel<128>;
    }
    return nullptr;
}

// Clusters of `kernel` that fit on the current device at once (0: none).
int fused_max_clusters(FusedKernel kernel, size_t smem) {
    if (!ensure_dynamic_smem(reinterpret_cast<const void *>(kernel), smem)) return 0;
    if (cudaFuncSetAttribute(reinterpret_cast<const void *>(kernel), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCs, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCs;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return n;
}

}  // namespace

bool router_fused_supported(const dmr_router_cfg_t &c, int B, int L) {
    if (!fused_kernel(c.d / c.heads) || B > 1024 || L > 128) return false;
    if ((long long)B * L > kRouterFusedMaxTokens) return false;
    return fused_plan(c, B, L).smem <= 227 * 1024;
}

// What either way takes, us.  A cluster takes its tokens in blocks of 32, and a block's steps through a layer cost about 28 us and 20 us per
// million of the layer's weights, whatever the chip could do at once; a layer's kernels cost about their sums' length in launches and latency
// and then 38 TFLOP/s of ALL tokens, the padded ones too.  Measured, one launch against layer by layer: d = 384, ffn 1536, 8 layers: 1024 tokens 2069 /
// 1890, 2048 of which half are padding 2150 / 2892, none 4066; d = 96, ffn 96, 12 layers: 256 tokens 497 / 592, 512 tokens 815 / 613, 4096
// 5568 / 937; d = 64, ffn 128, 2 layers: 512 tokens 102 / 107, 1024 tokens 167 / 118.
struct FusedCost {
    double layered, base, per_work;  // layer by layer; one launch: base + per_work * router_work()
};
FusedCost fused_cost(const dmr_router_cfg_t &c, long long T, int clusters) {
    const double d = c.d, f = c.ffn, weights = (4.0 * d * d + 2.0 * d * f) * 1e-6;  // of a layer, millions
    return {8.0 + c.layers * (30.0 + 0.055 * (3.0 * d + f) + (double)T * weights / 19.0), 20.0 + c.layers * (9.5 + 5.5 * weights),
            (28.0 + 20.0 * weights) / (kTokBlock * clusters)};
}

// ws: H [T][d], then two buffers of QKV [T][3 d]; the words at its end.
dmr_status_t launch_router_fused(const float *params, const dmr_router_cfg_t &c, const float *Z, const int32_t *lengths, int B, int L,
                                 float *probs, float *scores, int score_class, float *ws, const int32_t **done, cudaStream_t st) {
    *done = nullptr;
    FusedPlan p = fused_plan(c, B, L);
    FusedArgs &a = p.a;
    const size_t T = (size_t)B * L;
    a.params = params;
    a.Z = Z;
    a.lengths = lengths;
    a.probs = probs;
    a.scores = scores;
    a.score_class = score_class;
    a.H = ws;
    a.QKV = ws + T * c.d;
    a.counter = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(ws) + router_workspace_bytes(c, B, L) - kRouterWordBytes);
    FusedKernel kernel = fused_kernel(a.dh);
    static std::atomic<int> max_clusters[64][4];  // per device and kernel, at the largest shared memory: 0 = not asked yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return DMR_ERR_CUDA;
    std::atomic<int> &known = max_clusters[dev][a.dh == 16 ? 0 : a.dh == 32 ? 1 : a.dh == 64 ? 2 : 3];
    int most = known.load();
    if (most == 0) {
        most = fused_max_clusters(kernel, 227 * 1024);
        if (most < 1) return DMR_ERR_UNSUPPORTED;
        known.store(most);
    }
    const FusedCost cost = fused_cost(c, (long long)T, most);
    a.limit = cost.layered > cost.base ? (long long)((cost.layered - cost.base) / cost.per_work) : 0;
    const bool sure = router_work(c.layers, (long long)T, B) <= a.limit;
    if (!sure) {
        // The lengths may decide, on the device: the kernels of the other way are enqueued behind this one and return at once where it has taken the
        // call.  That is worth their microsecond each where sequences of evenly spread lengths, half the work of full ones, gain a tenth.
        const long long even = router_work(c.layers, ((long long)T + B) / 2, B);
        if (even > a.limit || cost.base + cost.per_work * (double)even + 1.3 * (2 + 7 * c.layers) > 0.9 * cost.layered) return DMR_ERR_UNSUPPORTED;
    }
    int clusters = (int)((T + 3) / 4);  // a task meets four tokens at a time
    if (clusters > most) clusters = most;
    cudaError_t e = cudaMemsetAsync(a.counter, 0, kRouterWordBytes, st);
    if (e != cudaSuccess) return launch_failed(e);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * kCs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCs;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, kernel, a);
    if (e != cudaSuccess) return launch_failed(e);
    if (!sure) *done = reinterpret_cast<const int32_t *>(a.counter + 1);
    return check_launch();
}

}  // namespace dmr
