// Importance-query predictor forward (paper Sec. 3.1 "Query prediction", App. A "two-layer MLP with
// hidden size 512"; Table 6 fixes the shapes: bias-free linears, layer norm with weight and bias):
//     q = W2 . act(W1 . LN(h))          per decoded token h, once per producer layer,
// the step right before the selection path: its output is the q_imp of the producer's consumer layers.
//
// At decode batch sizes both linears are bound by reading their weights once (8 MB per producer for an 8B-shaped
// model) and, at a microsecond of HBM time, by the latencies around that.  Two launches: hidden units (layer norm folded
// in), then outputs written in the layout tb_select_topk reads.  bf16: tensor-core tiles with the weights as the left
// operand; fp32: one warp (pair) per output row, 16-byte loads, every token of the call against the row while it is in
// registers.  No context: weights and scratch belong to the caller.
#include <cooperative_groups.h>
#include <type_traits>

#include "tb_common.cuh"
#include "tb_internal.h"

namespace tb {

#ifdef TB_PHASE_TIMING
__device__ unsigned long long g_pred_ns[2][12][256];     // [hidden / out kernel][stamp][block], last launch
__device__ __forceinline__ void pred_stamp(int k, int i) {
    if (threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        const int b = blockIdx.x + gridDim.x * blockIdx.y;
        if (b < 256) g_pred_ns[k][i][b] = t;
    }
}
extern "C" int tb_debug_pred_ns(unsigned long long* out) { return (int)cudaMemcpyFromSymbol(out, g_pred_ns, sizeof(g_pred_ns)); }
#else
#define pred_stamp(k, i) ((void)0)
#endif

namespace {

constexpr int kPredThreads = 256;
constexpr int kPredWarps = kPredThreads / 32;
constexpr int kPredMaxTokens = 64;
constexpr int kTokChunk = 8;        // tokens whose accumulators a warp keeps while it walks a weight row
constexpr int kStageTok = 16;       // tokens whose hidden units the output kernel stages in shared memory at once

__device__ __forceinline__ float activate(float a, int act) {
    if (act == TB_ACT_GELU) return 0.5f * a * (1.f + erff(a * 0.70710678118654752f));
    if (act == TB_ACT_SILU) return a / (1.f + __expf(-a));
    return fmaxf(a, 0.f);
}

// hidden[t][j] = act( sum_c W1[j][c] * ((h[t][c] - mean_t) * rstd_t * ln_w[c] + ln_b[c]) )
// A block owns kPredWarps / 2 hidden units, two warps per unit (half of the channels each), so that an
// 8B-shaped layer (512 units x 4096 channels) spreads over 128 blocks and a warp's share of a row is
// eight 16-byte loads, issued four at a time.
template <typename T>
__global__ void __launch_bounds__(kPredThreads) predictor_hidden_kernel(const T* __restrict__ H, const T* __restrict__ ln_w,
                                                                        const T* __restrict__ ln_b, const T* __restrict__ W1,
                                                                        float* __restrict__ hidden, int n_tok, int E, int hid,
                                                                        float eps, int act) {
    constexpr int P = Elem<T>::kPer16;
    constexpr int kUnits = kPredWarps / 2;
    pdl_launch_dependents();                           // the output kernel may start fetching its weights
    __shared__ float s_mean[kPredMaxTokens], s_rstd[kPredMaxTokens];
    __shared__ float s_half[kUnits][kTokChunk];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_vec = E / P;

    // Layer-norm statistics: sums of (h - h[0]) and of its square in one pass (the shift keeps the
    // variance accurate when the token's mean is large against its spread).  Few tokens: the whole
    // block per token; many: one warp per token.
    __shared__ float s_part[kPredWarps][2];
    auto token_sums = [&](int t, int first, int stride, float& s1, float& s2) {
        const uint4* h4 = reinterpret_cast<const uint4*>(H + (size_t)t * E);
        const float shift = Elem<T>::to_f32(H[(size_t)t * E]);
        float f[P];
        s1 = s2 = 0.f;
        for (int v = first; v < n_vec; v += stride) {
            Elem<T>::unpack16(__ldg(h4 + v), f);
#pragma unroll
            for (int e = 0; e < P; ++e) {
                const float d = f[e] - shift;
                s1 += d, s2 = fmaf(d, d, s2);
            }
        }
        s1 = warp_sum(s1), s2 = warp_sum(s2);
        return shift;
    };
    auto publish = [&](int t, float shift, float s1, float s2) {
        const float m = s1 / (float)E;
        s_mean[t] = shift + m, s_rstd[t] = rsqrtf(fmaxf(s2 / (float)E - m * m, 0.f) + eps);
    };
    if (n_tok < kPredWarps) {
        for (int t = 0; t < n_tok; ++t) {
            float s1, s2;
            const float shift = token_sums(t, tid, kPredThreads, s1, s2);
            if (lane == 0) s_part[warp][0] = s1, s_part[warp][1] = s2;
            __syncthreads();
            if (tid == 0) {
                float a = 0.f, b = 0.f;
                for (int w = 0; w < kPredWarps; ++w) a += s_part[w][0], b += s_part[w][1];
                publish(t, shift, a, b);
            }
            __syncthreads();
        }
    } else {
        for (int t = warp; t < n_tok; t += kPredWarps) {
            float s1, s2;
            const float shift = token_sums(t, lane, 32, s1, s2);
            if (lane == 0) publish(t, shift, s1, s2);
        }
        __syncthreads();
    }

    const int unit = warp >> 1, half = warp & 1;
    const int j = blockIdx.x * kUnits + unit;          // this warp pair's hidden unit
    const bool live = j < hid;
    const int v_begin = half * (n_vec / 2), v_end = half ? n_vec : n_vec / 2;
    const uint4* w4 = reinterpret_cast<const uint4*>(W1 + (size_t)(live ? j : 0) * E);
    const uint4* g4 = reinterpret_cast<const uint4*>(ln_w);
    const uint4* b4 = reinterpret_cast<const uint4*>(ln_b);
    for (int t0 = 0; t0 < n_tok; t0 += kTokChunk) {
        float acc[kTokChunk], mean[kTokChunk], rstd[kTokChunk];
#pragma unroll
        for (int u = 0; u < kTokChunk; ++u) {
            acc[u] = 0.f;
            const int t = min(t0 + u, n_tok - 1);
            mean[u] = s_mean[t], rstd[u] = s_rstd[t];
        }
        for (int v0 = v_begin + lane; v0 < v_end; v0 += 4 * 32) {   // four rounds of loads in flight
            uint4 wv[4], gv[4], bv[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int v = min(v0 + r * 32, v_end - 1);
                wv[r] = __ldg(w4 + v), gv[r] = __ldg(g4 + v), bv[r] = __ldg(b4 + v);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int v = v0 + r * 32;
                if (v >= v_end) break;
                float w[P], g[P], b[P];
                Elem<T>::unpack16(wv[r], w);
                Elem<T>::unpack16(gv[r], g);
                Elem<T>::unpack16(bv[r], b);
#pragma unroll
                for (int u = 0; u < kTokChunk; ++u) {
                    const int t = t0 + u;
                    if (t >= n_tok) break;             // uniform
                    float h[P];
                    Elem<T>::unpack16(__ldg(reinterpret_cast<const uint4*>(H + (size_t)t * E) + v), h);
#pragma unroll
                    for (int e = 0; e < P; ++e) acc[u] = fmaf(w[e], fmaf((h[e] - mean[u]) * rstd[u], g[e], b[e]), acc[u]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kTokChunk; ++u) acc[u] = warp_sum(acc[u]);
        if (half == 1 && lane == 0)
#pragma unroll
            for (int u = 0; u < kTokChunk; ++u) s_half[unit][u] = acc[u];
        __syncthreads();
        if (half == 0 && lane == 0 && live)
#pragma unroll
            for (int u = 0; u < kTokChunk; ++u)
                if (t0 + u < n_tok) hidden[(size_t)(t0 + u) * hid + j] = activate(acc[u] + s_half[unit][u], act);
        __syncthreads();
    }
}

// q_imp[slot][t][head][i] = sum_j W2[(slot, head, i)][j] * hidden[t][j]
template <typename T>
__global__ void __launch_bounds__(kPredThreads) predictor_out_kernel(const T* __restrict__ W2, const float* __restrict__ hidden,
                                                                     float* __restrict__ q_imp, int n_tok, int hid, int n_out,
                                                                     int per_slot, int stage_tok) {
    constexpr int P = Elem<T>::kPer16;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int o_raw = blockIdx.x * kPredWarps + warp;  // this warp's output row
    const bool live = o_raw < n_out;                   // idle warps still take part in the barriers
    const int o = live ? o_raw : 0;
    const uint4* w4 = reinterpret_cast<const uint4*>(W2 + (size_t)o * hid);
    const int n_vec = hid / P;
    const int slot = o / per_slot, within = o % per_slot;   // per_slot = heads * d'
    // The row's first vectors do not depend on the hidden units: fetch them while the kernel that
    // computes those is still running (programmatic dependent launch), then wait for it.
    constexpr int kPre = 2;                            // covers a 512-wide bf16 row
    uint4 pre[kPre];
#pragma unroll
    for (int r = 0; r < kPre; ++r) pre[r] = lane + 32 * r < n_vec ? __ldg(w4 + lane + 32 * r) : make_uint4(0u, 0u, 0u, 0u);
    pdl_wait();
    extern __shared__ float s_hidden[];                // stage_tok rows of `hid` floats
    for (int t0 = 0; t0 < n_tok; t0 += kTokChunk) {
        const int nt = min(kTokChunk, n_tok - t0);
        if (t0 % stage_tok == 0) {                     // (stage_tok is a multiple of kTokChunk)
            const int ns = min(stage_tok, n_tok - t0);
            __syncthreads();                           // the previous tokens are no longer read
            for (int i = threadIdx.x * 4; i < ns * hid; i += kPredThreads * 4)
                *reinterpret_cast<float4*>(s_hidden + i) = __ldcg(reinterpret_cast<const float4*>(hidden + (size_t)t0 * hid + i));
            __syncthreads();
        }
        const float* s_tok = s_hidden + (size_t)(t0 % stage_tok) * hid;
        float acc[kTokChunk];
#pragma unroll
        for (int u = 0; u < kTokChunk; ++u) acc[u] = 0.f;
        auto use = [&](int v, const uint4& wv) {
            float w[P];
            Elem<T>::unpack16(wv, w);
#pragma unroll
            for (int u = 0; u < kTokChunk; ++u) {
                if (u >= nt) break;                    // uniform
                const float* hp = s_tok + u * hid + v * P;
#pragma unroll
                for (int e = 0; e < P; e += 4) {
                    const float4 x = *reinterpret_cast<const float4*>(hp + e);
                    acc[u] = fmaf(w[e], x.x, acc[u]), acc[u] = fmaf(w[e + 1], x.y, acc[u]);
                    acc[u] = fmaf(w[e + 2], x.z, acc[u]), acc[u] = fmaf(w[e + 3], x.w, acc[u]);
                }
            }
        };
#pragma unroll
        for (int r = 0; r < kPre; ++r)
            if (lane + 32 * r < n_vec) use(lane + 32 * r, pre[r]);
        for (int v = lane + 32 * kPre; v < n_vec; v += 32) use(v, __ldg(w4 + v));
#pragma unroll
        for (int u = 0; u < kTokChunk; ++u) {
            const float a = warp_sum(acc[u]);
            if (lane == 0 && live && t0 + u < n_tok) q_imp[((size_t)slot * n_tok + (t0 + u)) * per_slot + within] = a;
        }
    }
}

// ---- bf16: both linears on the tensor cores, weights as the left operand ------------------------------
// D[32 weight rows x tokens] += W[32 x K] . X[K x tokens] with mma.sync.m16n8k16: the weights are exact in bf16, and
// the fp32 right operand (scaled hidden states, resp. hidden units) is split into bf16 terms, one MMA each, accumulated
// in fp32: three terms, which hold all 24 bits of it, for up to four tokens and for odd shapes (in groups of eight tokens),
// two (16 bits) for the rest.  A block's work is 32 weight rows x 512 channels -- 32 KB of
// weights, about what an SM receives in a memory latency, so that an 8B-shaped linear (8 MB) is 128 blocks that
// request everything they need at once -- against all tokens of the call.  The tensor pipe is idle most of the time
// and latency is what there is to save: every thread's weights are in flight before it looks at the tokens.
// Measured, one call of a 4096 -> 512 -> 4096 predictor in a chain of them: 7.2 us with 1 token, 7.2 with 8, 8.0 with 16, 11.0
// with 24, 14.1 with 47, 23 with 64, of which 1.3 are the weights at the copy bandwidth.  (With the token groups one after the
// other in the same blocks, as large as 32: 9.5 with 16, 12.0 with 24, 20.6 with 47, 31 with 64.)  The weights go through shared
// memory because their copies then cost no registers: with the fragments loaded straight into registers the kernels
// spilled and ran at 11.3 us.  Two blocks must fit an SM (they do up to 24 tokens): the output kernel's blocks sit beside the hidden kernel's and
// have their weights before the hidden units exist, and at one block per SM only 15 of the 16 clusters start at once.
//
// The 16 k-indices of an MMA step are mapped to channels so that every thread's operands are 16 contiguous bytes:
// over a run of 32 channels, thread (row gid, column pair tig) takes channels 8 tig .. 8 tig + 7; the first four feed
// the first MMA step (k = 2 tig, 2 tig + 1, 2 tig + 8, 2 tig + 9), the last four the second.  Both operands use the
// same mapping, so the sum over channels is unchanged.
constexpr int kTileRows = 32;        // weight rows of a block
constexpr int kChunk = 512;          // channels of a block's tile: 4 warps x 4 runs of 32, for each of two 16-row halves
constexpr int kTileTokMax = 24;      // tokens of a group; a kernel instance takes 8 * kN8 of them
constexpr int kXPitch = kChunk * 2 + 64;   // bytes per (term, token) row: eight rows' 64-byte pieces hit all banks twice
constexpr int kClusterK = 8;         // blocks (one cluster) that share the channels of a hidden-unit tile

__device__ __forceinline__ void mma_bf16_16x8x16(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Writes 8 consecutive values as bf16 terms, 16 bytes each, `stride` bytes apart.
template <int kTerms>
__device__ __forceinline__ void store_terms(unsigned char* dst, size_t stride, float* x) {
#pragma unroll
    for (int k = 0; k < kTerms; ++k) {
        uint32_t t[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const __nv_bfloat162 v = __floats2bfloat162_rn(x[e], x[e + 1]);
            t[e / 2] = *reinterpret_cast<const uint32_t*>(&v);
            x[e] -= __low2float(v), x[e + 1] -= __high2float(v);
        }
        *reinterpret_cast<uint4*>(dst + k * stride) = make_uint4(t[0], t[1], t[2], t[3]);
    }
}

// The block's weights of one chunk go to shared memory by 16-byte asynchronous copies, whole lines at a time; a warp
// then multiplies 16 of the rows (half mt) by a quarter kq of the 512 channels.
constexpr int kWBytes = kTileRows * kXPitch;
// requests channels [c_begin, min(c_begin + kChunk, c_end)) of rows row0 ..; rows past the matrix repeat its last one,
// channels past the end are zero
__device__ __forceinline__ void request_weights(unsigned char* ws, const __nv_bfloat16* __restrict__ W, int n_rows, int pitch, int row0,
                                                int c_begin, int c_end) {
#pragma unroll
    for (int i = 0; i < kTileRows * (kChunk / 8) / kPredThreads; ++i) {
        const int e = i * kPredThreads + threadIdx.x, row = e / (kChunk / 8), v = e % (kChunk / 8), c = c_begin + v * 8;
        unsigned char* dst = ws + row * kXPitch + v * 16;
        if (c < c_end)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(W + (size_t)min(row0 + row, n_rows - 1) * pitch + c) : "memory");
        else
            *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void wait_weights() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// acc += W . X for kN8 groups of eight staged tokens.  A single group has two accumulators, so that the chain of
// dependent MMAs is half as long.  kNorm: also gb += W . (column 0 = ln_w, column 1 = ln_b), whose operand gbx comes
// straight from the parameters.
template <int kN8>
constexpr int kAccs = kN8 == 1 ? 2 : kN8;
template <int kTerms, int kN8, bool kNorm>
__device__ __forceinline__ void mma_tile(float (&acc)[kAccs<kN8>][4], const unsigned char* ws, const unsigned char* xs, float* gb,
                                         const uint4* gbx) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gid = lane >> 2, tig = lane & 3, mt = warp >> 2, kq = warp & 3;
    const int off = (kq * 128 + 8 * tig) * 2;
    const unsigned char* wa = ws + (mt * 16 + gid) * kXPitch + off;
    const unsigned char* x0 = xs + gid * kXPitch + off;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint4 a = *reinterpret_cast<const uint4*>(wa + r * 64), b = *reinterpret_cast<const uint4*>(wa + 8 * kXPitch + r * 64);
        if constexpr (kNorm) {
            mma_bf16_16x8x16(gb, a.x, b.x, a.y, b.y, gbx[r].x, gbx[r].y);
            mma_bf16_16x8x16(gb, a.z, b.z, a.w, b.w, gbx[r].z, gbx[r].w);
        }
#pragma unroll
        for (int k = 0; k < kTerms; ++k) {
            uint4 x[kN8];
#pragma unroll
            for (int n = 0; n < kN8; ++n) x[n] = *reinterpret_cast<const uint4*>(x0 + (k * kN8 + n) * 8 * kXPitch + r * 64);
#pragma unroll
            for (int n = 0; n < kN8; ++n) mma_bf16_16x8x16(acc[n], a.x, b.x, a.y, b.y, x[n].x, x[n].y);
#pragma unroll
            for (int n = 0; n < kN8; ++n) mma_bf16_16x8x16(acc[kN8 == 1 ? 1 : n], a.z, b.z, a.w, b.w, x[n].z, x[n].w);
        }
    }
}
// The four channel quarters' accumulators, [quarter][row][token]
template <int kN8>
using TileSums = float[4][kTileRows][kN8 * 8 + 1];
template <int kN8>
__device__ __forceinline__ void put_sums(TileSums<kN8>& s, float (&acc)[kAccs<kN8>][4]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gid = lane >> 2, tig = lane & 3, row = (warp >> 2) * 16 + gid;
    if constexpr (kN8 == 1) acc[0][0] += acc[1][0], acc[0][1] += acc[1][1], acc[0][2] += acc[1][2], acc[0][3] += acc[1][3];
#pragma unroll
    for (int n = 0; n < kN8; ++n) {
        s[warp & 3][row][n * 8 + 2 * tig] = acc[n][0], s[warp & 3][row][n * 8 + 2 * tig + 1] = acc[n][1];
        s[warp & 3][row + 8][n * 8 + 2 * tig] = acc[n][2], s[warp & 3][row + 8][n * 8 + 2 * tig + 1] = acc[n][3];
    }
}
template <int kN8>
__device__ __forceinline__ float get_sum(const TileSums<kN8>& s, int row, int tok) { return (s[0][row][tok] + s[1][row][tok]) + (s[2][row][tok] + s[3][row][tok]); }

// hidden[t][j] = act( sum_c W1[j][c] * ((h[t][c] - mean_t) * rstd_t * ln_w[c] + ln_b[c]) ), fp32 or (two terms) as
// bf16 [term][t][j], for 32 hidden units per cluster of eight blocks, an eighth of the channels each.  No block waits for a token's statistics: with a shift s of
// its own (the token's mean over the block's first channels) block b computes
//     P = sum_c w ln_w (h - s),   G = sum_c w ln_w,   B = sum_c w ln_b
// and the shifted sums of h and h^2 over its channels; behind one exchange through distributed shared memory
//     sum = rstd * sum_b (P_b - (mean - s_b) G_b) + sum_b B_b
// where mean - s_b is small against the spread, so nothing cancels.  Blocks are summed in rank order.
template <int kTerms, int kN8, int kPerSm>
__global__ void __launch_bounds__(kPredThreads, kPerSm) predictor_hidden_tile_kernel(const __nv_bfloat16* __restrict__ H,
                                                                                const __nv_bfloat16* __restrict__ ln_w,
                                                                                const __nv_bfloat16* __restrict__ ln_b,
                                                                                const __nv_bfloat16* __restrict__ W1,
                                                                                float* __restrict__ hidden, int n_tok, int E, int hid,
                                                                                float eps, int act) {
    namespace cg = cooperative_groups;
    using EB = Elem<__nv_bfloat16>;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();        // == blockIdx.x
    constexpr int kRows = kTileRows / kClusterK;       // hidden units this block finishes
    constexpr int kTileTok = kN8 * 8, kOwn = kN8;      // tokens of a group; of those, the ones a warp looks after
    constexpr size_t kTermStride = (size_t)kTileTok * kXPitch;
    extern __shared__ __align__(128) unsigned char ws[];   // weights [32 rows][kXPitch], then states [term][token][kXPitch]
    unsigned char* xs = ws + kWBytes;
    __shared__ TileSums<kN8> s_sum;
    __shared__ float2 s_gb[4][kTileRows];              // (G, B) of the block's rows, per channel quarter
    // from every block of the cluster: P and (G, B) of this block's rows, and every token's (shift, shifted sum, shifted sum of squares)
    __shared__ float s_p[kClusterK][kRows][kTileTok];
    __shared__ float2 s_gb_all[kClusterK][kRows];
    __shared__ float4 s_stat[kClusterK][kTileTok];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gid = lane >> 2, tig = lane & 3;
    const int j0 = blockIdx.y * kTileRows;
    const int span = (((E + 31) / 32 + kClusterK - 1) / kClusterK) * 32;     // channels of a block
    const int c_begin = min(E, rank * span), c_end = min(E, c_begin + span);
    const int n_chunk = (span + kChunk - 1) / kChunk;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    pred_stamp(0, 0);
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");    // awaited before the first remote write: the block runs
    // The states may come from the predecessor, and so may the weights: wait, then let the output kernel get ready.
    pdl_wait();
    pdl_launch_dependents();
    pred_stamp(0, 1);

    const int t0 = blockIdx.z * kTileTok, n_here = min(kTileTok, n_tok - t0);   // this cluster's tokens
    {
        float acc[kAccs<kN8>][4] = {}, gb[4] = {};
        float shift[kOwn], s1[kOwn], s2[kOwn];
#pragma unroll
        for (int i = 0; i < kOwn; ++i) shift[i] = s1[i] = s2[i] = 0.f;
        for (int kc = 0; kc < n_chunk; ++kc) {
            const int c0 = c_begin + kc * kChunk;
            if (kc) __syncthreads();                   // the previous chunk's operands have been read
            request_weights(ws, W1, hid, E, j0, c0, c_end);
            // A warp looks after tokens warp, warp + 8, ... of the group, a lane after channels 8 lane .. + 7 and
            // 256 + 8 lane .. + 7 of the chunk.
            uint4 hv[kOwn][2], gv[2];
#pragma unroll
            for (int i = 0; i < kOwn; ++i)
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const int tl = i * kPredWarps + warp, c = c0 + v * 256 + lane * 8;
                    hv[i][v] = tl < n_here && c < c_end ? __ldg(reinterpret_cast<const uint4*>(H + (size_t)(t0 + tl) * E + c)) : zero;
                }
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                const int c = c0 + v * 256 + lane * 8;
                gv[v] = c < c_end ? __ldg(reinterpret_cast<const uint4*>(ln_w + c)) : zero;
            }
            // right operand of the G, B product: column 0 = layer-norm weights, column 1 = biases
            uint4 gbx[4];
            const __nv_bfloat16* src = gid == 0 ? ln_w : ln_b;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int c = c0 + ((warp & 3) * 4 + r) * 32 + 8 * tig;
                gbx[r] = gid < 2 && c < c_end ? __ldg(reinterpret_cast<const uint4*>(src + c)) : zero;
            }
            if (kc == 0) {
                const int n = min(kChunk, c_end - c0);
#pragma unroll
                for (int i = 0; i < kOwn; ++i) {
                    float f[8];
                    EB::unpack16(hv[i][0], f);
                    shift[i] = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]));
                    EB::unpack16(hv[i][1], f);
                    shift[i] += ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < kOwn; ++i) shift[i] += __shfl_xor_sync(0xffffffffu, shift[i], o);
#pragma unroll
                for (int i = 0; i < kOwn; ++i) shift[i] = n > 0 ? shift[i] / (float)n : 0.f;
            }
#pragma unroll
            for (int i = 0; i < kOwn; ++i) {
                const int tl = i * kPredWarps + warp;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const bool in = c0 + v * 256 + lane * 8 < c_end;
                    float h[8], g[8];
                    EB::unpack16(hv[i][v], h), EB::unpack16(gv[v], g);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float d = in ? h[e] - shift[i] : 0.f;      // (tokens past the end: all zero)
                        s1[i] += d, s2[i] = fmaf(d, d, s2[i]);
                        h[e] = d * g[e];
                    }
                    store_terms<kTerms>(xs + (size_t)tl * kXPitch + (v * 256 + lane * 8) * 2, kTermStride, h);
                }
            }
            pred_stamp(0, 7);
            wait_weights();
            __syncthreads();
            pred_stamp(0, 2);
            mma_tile<kTerms, kN8, true>(acc, ws, xs, gb, gbx);
        }
        put_sums<kN8>(s_sum, acc);
        if (tig == 0) {
            s_gb[warp & 3][(warp >> 2) * 16 + gid] = make_float2(gb[0], gb[1]);
            s_gb[warp & 3][(warp >> 2) * 16 + gid + 8] = make_float2(gb[2], gb[3]);
        }
        __syncthreads();
        pred_stamp(0, 3);
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        for (int e = tid; e < kTileRows * kTileTok; e += kPredThreads) {
            const int row = e / kTileTok, tok = e % kTileTok;
            if (tok < n_here) *cluster.map_shared_rank(&s_p[rank][row % kRows][tok], row / kRows) = get_sum<kN8>(s_sum, row, tok);
        }
        if (tid < kTileRows) {
            const float2 a = s_gb[0][tid], b = s_gb[1][tid], c = s_gb[2][tid], d = s_gb[3][tid];
            *cluster.map_shared_rank(&s_gb_all[rank][tid % kRows], tid / kRows) = make_float2((a.x + b.x) + (c.x + d.x), (a.y + b.y) + (c.y + d.y));
        }
#pragma unroll
        for (int i = 0; i < kOwn; ++i) {
            const int tl = i * kPredWarps + warp;
            if (tl >= n_here) break;                   // warp-uniform
            const float a = warp_sum(s1[i]), b = warp_sum(s2[i]);
            if (lane < kClusterK) *cluster.map_shared_rank(&s_stat[rank][tl], lane) = make_float4(shift[i], a, b, 0.f);   // lane r tells block r
        }
        pred_stamp(0, 4);
        cluster.sync();
        pred_stamp(0, 5);
        if (tid < kRows * kTileTok) {
            const int row = tid / kTileTok, tok = tid % kTileTok, j = j0 + rank * kRows + row;
            if (tok < n_here && j < hid) {
                float4 st[kClusterK];
                float mean = 0.f;
#pragma unroll
                for (int r = 0; r < kClusterK; ++r) {
                    st[r] = s_stat[r][tok];
                    const float n = (float)max(0, min(span, E - r * span));
                    mean += fmaf(n, st[r].x, st[r].y);
                }
                mean /= (float)E;
                float var = 0.f, sum = 0.f, bias = 0.f;
#pragma unroll
                for (int r = 0; r < kClusterK; ++r) {
                    // sum of (h - mean)^2 = sum of (d - u)^2 with d = h - shift, u = mean - shift
                    const float n = (float)max(0, min(span, E - r * span)), u = mean - st[r].x;
                    const float2 w = s_gb_all[r][row];
                    var += fmaf(u, fmaf(n, u, -2.f * st[r].y), st[r].z);
                    sum += fmaf(-u, w.x, s_p[r][row][tok]);
                    bias += w.y;
                }
                const float rstd = rsqrtf(fmaxf(var / (float)E, 0.f) + eps);
                const float x = activate(fmaf(rstd, sum, bias), act);
                if constexpr (kTerms == 2) {           // two terms take the room of the fp32 value: split here, once
                    __nv_bfloat16* term = reinterpret_cast<__nv_bfloat16*>(hidden) + (size_t)(t0 + tok) * hid + j;
                    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
                    term[0] = hi, term[(size_t)n_tok * hid] = __float2bfloat16_rn(x - __bfloat162float(hi));
                } else {
                    hidden[(size_t)(t0 + tok) * hid + j] = x;
                }
            }
        }
        pred_stamp(0, 6);
    }
}

// q_imp for 32 output rows per block, all hidden units.
template <int kTerms, int kN8, int kPerSm>
__global__ void __launch_bounds__(kPredThreads, kPerSm) predictor_out_tile_kernel(const __nv_bfloat16* __restrict__ W2, const float* __restrict__ hidden,
                                                                          float* __restrict__ q_imp, int n_tok, int hid, int n_out,
                                                                          int per_slot) {
    extern __shared__ __align__(128) unsigned char ws[];   // weights [32 rows][kXPitch], then hidden units [term][token][kXPitch]
    unsigned char* xs = ws + kWBytes;
    constexpr int kTileTok = kN8 * 8;
    constexpr size_t kTermStride = (size_t)kTileTok * kXPitch;
    __shared__ TileSums<kN8> s_sum;
    const int tid = threadIdx.x;
    const int o0 = blockIdx.x * kTileRows, n_chunk = (hid + kChunk - 1) / kChunk;
    // the weights do not depend on the hidden units (and the predecessor, which computes those, started after
    // everything before it): fetch them, then wait
    pred_stamp(1, 0);
    request_weights(ws, W2, n_out, hid, o0, 0, hid);
    pdl_wait();
    pdl_launch_dependents();
    pred_stamp(1, 1);
    const int t0 = blockIdx.y * kTileTok, n_here = min(kTileTok, n_tok - t0);   // this block's tokens
    {
        float acc[kAccs<kN8>][4] = {};
        for (int kc = 0; kc < n_chunk; ++kc) {
            if (kc) {
                __syncthreads();                       // the previous chunk's operands have been read
                request_weights(ws, W2, n_out, hid, o0, kc * kChunk, hid);
            }
            constexpr int kVec = kChunk / 8, kStep = kPredThreads / kVec;      // 8 values at a time, four tokens per round
            const int c = kc * kChunk + tid % kVec * 8;
            if constexpr (kTerms == 2) {               // the hidden-unit kernel has split them
#pragma unroll
                for (int i = 0; i < kTerms * kTileTok / kStep; ++i) {
                    const int row = i * kStep + tid / kVec, tl = row % kTileTok;
                    unsigned char* dst = xs + row * kXPitch + tid % kVec * 16;
                    if (tl < n_here && c < hid)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)),
                                     "l"(reinterpret_cast<const __nv_bfloat16*>(hidden) + ((size_t)(row / kTileTok) * n_tok + t0 + tl) * hid + c)
                                     : "memory");
                    else
                        *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            } else {
                float4 x[kTileTok / kStep][2];
#pragma unroll
                for (int i = 0; i < kTileTok / kStep; ++i) {
                    const int tl = i * kStep + tid / kVec;
                    const bool in = tl < n_here && c < hid;
                    const float4* src = reinterpret_cast<const float4*>(hidden + (size_t)(t0 + tl) * hid + c);
                    x[i][0] = in ? __ldcg(src) : make_float4(0.f, 0.f, 0.f, 0.f);
                    x[i][1] = in ? __ldcg(src + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int i = 0; i < kTileTok / kStep; ++i) {
                    float v[8] = {x[i][0].x, x[i][0].y, x[i][0].z, x[i][0].w, x[i][1].x, x[i][1].y, x[i][1].z, x[i][1].w};
                    store_terms<kTerms>(xs + (size_t)(i * kStep + tid / kVec) * kXPitch + tid % kVec * 16, kTermStride, v);
                }
            }
            wait_weights();
            __syncthreads();
            pred_stamp(1, 3);
            mma_tile<kTerms, kN8, false>(acc, ws, xs, nullptr, nullptr);
        }
        put_sums<kN8>(s_sum, acc);
        __syncthreads();
        pred_stamp(1, 4);
        for (int e = tid; e < kTileRows * kTileTok; e += kPredThreads) {
            const int row = e % kTileRows, tok = e / kTileRows, o = o0 + row;
            if (tok < n_here && o < n_out) q_imp[((size_t)(o / per_slot) * n_tok + t0 + tok) * per_slot + o % per_slot] = get_sum<kN8>(s_sum, row, tok);
        }
    }
    pred_stamp(1, 5);
}

}  // namespace

}  // namespace tb

extern "C" tb_status tb_predict_importance_queries(const tb_predictor* p, const void* hidden_dev, int32_t n_tokens,
                                                   float* scratch_dev, float* q_imp_dev, void* stream) {
    using namespace tb;
    if (!p || !hidden_dev || !scratch_dev || !q_imp_dev || !p->ln_weight || !p->ln_bias || !p->w1 || !p->w2) return TB_ERR_INVALID_ARG;
    if (p->dtype != TB_F32 && p->dtype != TB_BF16) return TB_ERR_INVALID_ARG;
    if (n_tokens <= 0 || p->model_dim <= 0 || p->hidden_dim <= 0 || p->n_q_heads <= 0 || p->n_slots <= 0 || p->imp_dim <= 0 ||
        !(p->ln_eps >= 0.f))
        return TB_ERR_INVALID_ARG;
    if (p->activation != TB_ACT_GELU && p->activation != TB_ACT_SILU && p->activation != TB_ACT_RELU) return TB_ERR_INVALID_ARG;
    if (n_tokens > kPredMaxTokens) return TB_ERR_CAPACITY;
    const int per16 = p->dtype == TB_BF16 ? 8 : 4;     // rows are read 16 bytes at a time
    if (p->model_dim % per16 || p->hidden_dim % per16 || p->hidden_dim > 1536) return TB_ERR_UNSUPPORTED;
    const uintptr_t align = (uintptr_t)hidden_dev | (uintptr_t)p->ln_weight | (uintptr_t)p->ln_bias | (uintptr_t)p->w1 |
                            (uintptr_t)p->w2 | (uintptr_t)scratch_dev;
    if (align & 15) return TB_ERR_INVALID_ARG;
    const long long n_out = (long long)p->n_slots * p->n_q_heads * p->imp_dim;
    if (n_out > (1ll << 24)) return TB_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    const int per_slot = p->n_q_heads * p->imp_dim, n_out_i = (int)n_out;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kPredThreads, 1, 1), cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see pdl_wait()
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = kClusterK, attr[1].val.clusterDim.y = 1, attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cudaError_t e;
    if (p->dtype == TB_BF16) {
        // The tokens go to the clusters (blocks) of grid layers in groups of 8, 16 or 24, the smallest for which the hidden kernel
        // still runs at once: the preparation of a group is what its blocks' time grows with, and more groups read the weights
        // from L2.  Otherwise as few groups as hold 24.  us per call, 4096 -> 512 -> 4096, groups of 8 / 16 / 24: 16 tokens 7.8 /
        // 9.5 / 9.5, 24 10.7 / 11.8 / 11.8, 32 15 / 10.8 / 13.3, 47 19 / 18.4 / 13.3; with 1024 hidden units, twice the blocks, 32
        // tokens 27 / 21.4 / 23.3, 64 48 / 38.6 / 33.9.
        // Groups of eight come compiled for two and for three blocks per SM.  The third costs registers (80 a thread) and is taken
        // only where two per SM do not hold the grid: 5120 -> 512, 9 to 16 tokens 10.1-10.4 us with two, 12.1 as one group of 16.
        int n8 = 1;
        bool two_per_sm = true;
        if (n_tokens > 8) {
            static std::atomic<int> sm_counts[64];
            int dev = 0, sms = 0;
            if (cudaGetDevice(&dev) != cudaSuccess) return TB_ERR_CUDA;
            if (dev < 64) sms = sm_counts[dev].load(std::memory_order_relaxed);
            if (!sms && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return TB_ERR_CUDA;
            if (dev < 64) sm_counts[dev].store(sms, std::memory_order_relaxed);
            const int tiles = kClusterK * ((p->hidden_dim + kTileRows - 1) / kTileRows);
            auto blocks = [&](int eights) { return tiles * ((n_tokens + 8 * eights - 1) / (8 * eights)); };
            n8 = blocks(1) <= 3 * sms ? 1 : blocks(2) <= 2 * sms ? 2 : 3;
            if (n8 == 3 && blocks(3) > 2 * sms) {
                const int groups = (n_tokens + kTileTokMax - 1) / kTileTokMax;
                n8 = ((n_tokens + groups - 1) / groups + 7) / 8;
            }
            two_per_sm = blocks(n8) <= 2 * sms;
        }
        auto launch = [&](auto terms, auto eights, auto per_sm) {
            constexpr int kTerms = decltype(terms)::value, kN8 = decltype(eights)::value, kPerSm = decltype(per_sm)::value;
            constexpr int smem = kWBytes + kTerms * kN8 * 8 * kXPitch;
            static DeviceFlags done;
            cudaError_t r = once_per_device(done, [&] {
                const cudaError_t e = cudaFuncSetAttribute(predictor_hidden_tile_kernel<kTerms, kN8, kPerSm>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
                return e != cudaSuccess ? e : cudaFuncSetAttribute(predictor_out_tile_kernel<kTerms, kN8, kPerSm>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            });
            if (r != cudaSuccess) return r;
            cfg.dynamicSmemBytes = smem;
            const unsigned n_groups = (unsigned)((n_tokens + kN8 * 8 - 1) / (kN8 * 8));
            cfg.gridDim = dim3(kClusterK, (p->hidden_dim + kTileRows - 1) / kTileRows, n_groups), cfg.numAttrs = 2;
            r = cudaLaunchKernelEx(&cfg, predictor_hidden_tile_kernel<kTerms, kN8, kPerSm>, (const __nv_bfloat16*)hidden_dev,
                                               (const __nv_bfloat16*)p->ln_weight, (const __nv_bfloat16*)p->ln_bias,
                                               (const __nv_bfloat16*)p->w1, scratch_dev, (int)n_tokens, (int)p->model_dim,
                                               (int)p->hidden_dim, p->ln_eps, (int)p->activation);
            if (r != cudaSuccess) return r;
            cfg.gridDim = dim3((unsigned)((n_out + kTileRows - 1) / kTileRows), n_groups, 1), cfg.numAttrs = 1;
            return cudaLaunchKernelEx(&cfg, predictor_out_tile_kernel<kTerms, kN8, kPerSm>, (const __nv_bfloat16*)p->w2, (const float*)scratch_dev,
                                      q_imp_dev, (int)n_tokens, (int)p->hidden_dim, n_out_i, per_slot);
        };
        using std::integral_constant;
        // 24 bits of both right operands for up to four tokens, and for shapes off the 32-channel runs (always computed so)
        const bool whole = n_tokens < 5 || p->model_dim % 32 || p->hidden_dim % 32 || n_out % 8;
        using I1 = integral_constant<int, 1>;
        using I2 = integral_constant<int, 2>;
        using I3 = integral_constant<int, 3>;
        if (whole) e = launch(I3{}, I1{}, I2{});
        else if (n8 == 1) e = two_per_sm ? launch(I2{}, I1{}, I2{}) : launch(I2{}, I1{}, I3{});
        else if (n8 == 2) e = launch(I2{}, I2{}, I2{});
        else e = launch(I2{}, I3{}, I2{});
    } else {
        const int g1 = (p->hidden_dim + kPredWarps / 2 - 1) / (kPredWarps / 2), g2 = (int)((n_out + kPredWarps - 1) / kPredWarps);
        int stage_tok = (int)(48 * 1024 / (p->hidden_dim * sizeof(float))) / kTokChunk * kTokChunk;   // hidden_dim <= 1536 gives >= 8
        stage_tok = stage_tok > kStageTok ? kStageTok : stage_tok < kTokChunk ? kTokChunk : stage_tok;
        predictor_hidden_kernel<float><<<g1, kPredThreads, 0, s>>>((const float*)hidden_dev, (const float*)p->ln_weight,
                                                                   (const float*)p->ln_bias, (const float*)p->w1, scratch_dev, n_tokens,
                                                                   p->model_dim, p->hidden_dim, p->ln_eps, p->activation);
        cfg.gridDim = dim3(g2, 1, 1), cfg.numAttrs = 1;
        cfg.dynamicSmemBytes = (size_t)stage_tok * p->hidden_dim * sizeof(float);
        e = cudaLaunchKernelEx(&cfg, predictor_out_kernel<float>, (const float*)p->w2, (const float*)scratch_dev, q_imp_dev,
                               (int)n_tokens, (int)p->hidden_dim, n_out_i, per_slot, stage_tok);
    }
    if (e != cudaSuccess) return TB_ERR_CUDA;
    return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}
