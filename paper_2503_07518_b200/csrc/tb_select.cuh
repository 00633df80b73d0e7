// Pieces shared by the selection kernels: the scoring arithmetic (FMA chains; bf16 rows also on the tensor
// cores, with exact products and fp32 sums in another order), launch-unit decoding, neighbours and lists.
#pragma once

#include <algorithm>
#include <type_traits>

#include "tb_common.cuh"
#include "tb_internal.h"

namespace tb {

// ---- scoring arithmetic shared by the standalone and the fused kernel --------------------------

// Importance query of KV head h: sum over the g query heads of the group, in head order.
template <int DP>
__device__ __forceinline__ void load_group_query(const float* __restrict__ q_imp_unit, int g, float* qr) {
#pragma unroll
    for (int j = 0; j < DP; ++j) qr[j] = 0.f;
    for (int u = 0; u < g; ++u)
#pragma unroll
        for (int j = 0; j < DP; ++j) qr[j] += q_imp_unit[u * DP + j];
}

// Dot product of one projected-key row (NCH 16-byte chunks fetched by `ld(c)`) with qr.  Two FMA
// chains (even / odd chunks), each in ascending element order, added at the end: the result depends
// only on the row's bytes, never on where the row sits.
template <typename T, int DP, typename LoadChunk>
__device__ __forceinline__ float row_score(const float* qr, LoadChunk ld) {
    constexpr int P = Elem<T>::kPer16;
    constexpr int NCH = DP / P;
    float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        uint4 v = ld(c);
        float f[P];
        Elem<T>::unpack16(v, f);
        if (c & 1) {
#pragma unroll
            for (int e = 0; e < P; ++e) acc1 = fmaf(qr[c * P + e], f[e], acc1);
        } else {
#pragma unroll
            for (int e = 0; e < P; ++e) acc0 = fmaf(qr[c * P + e], f[e], acc0);
        }
    }
    return acc0 + acc1;
}

// The same for TB_GROUP_MAX: the row's score is the largest of the g heads' dot products.  `qs` holds
// the g importance queries, [g][DP] floats in shared memory (every lane reads the same words: broadcast).
// Each head's dot product is accumulated exactly as in row_score.
template <typename T, int DP, typename LoadChunk>
__device__ __forceinline__ float row_score_max(const float* qs, int g, LoadChunk ld) {
    constexpr int P = Elem<T>::kPer16;
    constexpr int NCH = DP / P;
    float f[DP];
#pragma unroll
    for (int c = 0; c < NCH; ++c) Elem<T>::unpack16(ld(c), f + c * P);
    float best = -INFINITY;
    for (int u = 0; u < g; ++u) {
        const float4* q4 = reinterpret_cast<const float4*>(qs + u * DP);
        float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
#pragma unroll
            for (int e = 0; e < P; e += 4) {
                const float4 q = q4[(c * P + e) / 4];
                float& acc = (c & 1) ? acc1 : acc0;
                acc = fmaf(q.x, f[c * P + e], acc), acc = fmaf(q.y, f[c * P + e + 1], acc);
                acc = fmaf(q.z, f[c * P + e + 2], acc), acc = fmaf(q.w, f[c * P + e + 3], acc);
            }
        }
        best = fmaxf(best, acc0 + acc1);
    }
    return best;
}

// How a selection kernel scores a row under the reduction RED (TB_GROUP_SUM: one dot product with the
// summed query held in registers; TB_GROUP_MAX: g dot products against the queries in shared memory).
template <typename T, int DP, int RED>
struct GroupScorer {
    float qr[RED == TB_GROUP_SUM ? DP : 1];
    const float* qs;
    int g;
    // q_unit: the group's g queries [g][DP] in global memory; qs_smem: room for kMaxGroup * DP floats.
    // All threads of the block call it; with TB_GROUP_MAX a block barrier must follow before score().
    __device__ __forceinline__ void load(const float* __restrict__ q_unit, int g_, float* qs_smem) {
        g = g_, qs = qs_smem;
        if constexpr (RED == TB_GROUP_SUM) {
            load_group_query<DP>(q_unit, g_, qr);
        } else {
            for (int i = threadIdx.x; i < g_ * DP; i += blockDim.x) qs_smem[i] = q_unit[i];
        }
    }
    // The same from queries that already sit in shared memory ([g][DP] floats, visible to the thread):
    // the summed query is built in the same order, so the scores are the same bits.
    __device__ __forceinline__ void load_staged(const float* qs_smem, int g_) {
        g = g_, qs = qs_smem;
        if constexpr (RED == TB_GROUP_SUM) load_group_query<DP>(qs_smem, g_, qr);
    }
    template <typename LoadChunk>
    __device__ __forceinline__ float score(LoadChunk ld) const {
        if constexpr (RED == TB_GROUP_SUM) return row_score<T, DP>(qr, ld);
        else return row_score_max<T, DP>(qs, g, ld);
    }
};

// A selection unit is one index list: (layer, sequence, list head h < Hl).
__device__ __forceinline__ void decode_unit(const Geom& gm, const UnitTable& ut, int u, int& ll, int& s, int& h) {
    h = u % gm.Hl;
    s = (u / gm.Hl) % ut.n_seq;
    ll = u / (gm.Hl * ut.n_seq);
}
// Row of the unit in the context's lists, counts and parked-key workspace.
__device__ __forceinline__ size_t list_unit(const Geom& gm, const UnitTable& ut, int ll, int s, int h) {
    return ((size_t)(ut.layer_begin + ll) * gm.max_batch + ut.seq_id[s]) * gm.Hl + h;
}
// Key stream of the unit in the projected-key cache: its own (one list per KV head), its KV head's
// (one list per query head) or the layer's only one.
__device__ __forceinline__ size_t key_unit(const Geom& gm, const UnitTable& ut, int ll, int s, int h) {
    return ((size_t)(ut.layer_begin + ll) * gm.max_batch + ut.seq_id[s]) * gm.Hi + (h * gm.Hi) / gm.Hl;
}
// The unit's importance queries: gl consecutive rows of q_imp [layer_count][n_seq][Hl * gl][d'].
__device__ __forceinline__ size_t query_row(const Geom& gm, const UnitTable& ut, int ll, int s, int h) {
    return ((size_t)(ll * ut.n_seq + s) * gm.Hl + h) * gm.gl;
}

// With device-resident lengths the host cannot check, at replay time, that every candidate has a projected
// key: one thread per block does, and reports through the status word (the selection itself goes on).
__device__ __forceinline__ void check_candidates_projected(const Geom& gm, const UnitTable& ut, int ll, int s, int hi, int32_t* status) {
    if (ut.use_dev_len && threadIdx.x == 0) {
        const size_t pair = (size_t)(ut.layer_begin + ll) * gm.max_batch + ut.seq_id[s];
        if (ut.len_proj_dev[pair] < hi) atomicExch(status, kStatusUnprojected);
    }
}

// Launch order of the (layer, sequence) pairs: longest first, so that the blocks still running when
// the grid drains are the short ones.
struct WaveOrder {
    uint16_t pair[kMaxLaunchUnits];
};

// The pairs of a launch, longest first, and their candidates; returns the most.
inline int longest_first(const UnitTable& ut, const SelectArgs& a, WaveOrder& order, int (&cand)[kMaxLaunchUnits]) {
    const int n_pairs = ut.layer_count * ut.n_seq;
    for (int i = 0; i < n_pairs; ++i) {
        const int L = ut.len[i], lo = a.sinks < L ? a.sinks : L, hi = L - a.recent > lo ? L - a.recent : lo;
        cand[i] = hi - lo, order.pair[i] = (uint16_t)i;
    }
    std::stable_sort(order.pair, order.pair + n_pairs, [&](uint16_t x, uint16_t y) { return cand[x] > cand[y]; });
    return cand[order.pair[0]];
}

// Candidates of a problem whose kernel keeps something per candidate in shared memory.  A replayed graph may find a sequence
// longer than its launch was sized for (it outgrew the declared reserve): the candidates past `room` are left out and the
// status word says so.
__device__ __forceinline__ int candidates_within(int n, int room, int32_t* status) {
    if (n <= room) return n;
    if (threadIdx.x == 0) atomicExch(status, kStatusCapacity);
    return room;
}

// ---- bf16 rows straight into tensor-core fragments ------------------------------------------------------
//
// Over a 64-byte row (32 dimensions) thread tig of a row's four takes 16 contiguous bytes, so a warp's 16-byte load is
// eight whole rows, and with the query's dimensions permuted the same way the four 4-byte words are the A operand of two
// m16n8k16 steps (8 bytes and one step for 16 dimensions).  No shared memory, no barrier; every warp keeps kU groups of 32
// rows in flight.   D[16 rows x 8] += K[16 x 16] . Q[16 x 8], fp32 accumulators; Q is split into three bf16 terms that hold
// all 24 bits of the fp32 query, so every product is exact and only the fp32 sums round (against fp64, 32 dimensions, four
// heads: rms error 1.7e-8 of sum |q k|, where the FMA chains above have 2.5e-8; 16 dimensions 1.9e-8 and 2.5e-8).
// TB_GROUP_SUM: the columns are the terms of the summed query, (high, middle, low, 0) twice, so a group takes four MMAs and
// its operands four registers; a lane adds two terms, its neighbour the other two, one shuffle brings them together at the lane
// that owns the row.  (All eight columns the summed query, the terms one after the other: 12 MMAs at 8.7 cycles each in chains
// of six, operands from shared memory.)  TB_GROUP_MAX: column = head, the terms one after the other, lowest first; a row's
// score is the largest over the columns.  A row's score depends only on its bytes, never on where it sits.  Infinities do not
// survive the split (a query's lower terms are zero or of either sign: inf * 0, inf - inf): rows with an infinite score are
// scored again, by the FMA chains, behind the stream (rescore).  The kernels look for them only where a sum over the scores, or
// a query, is not finite.
constexpr int kQueryFrags = 3 * 2 * 32;   // TB_GROUP_MAX, a query's B fragments: terms x steps x lanes

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ bool is_finite(float s) { return fabsf(s) <= 3.402823466e38f; }
// row_score / row_score_max of one bf16 row in global memory, from the staged queries: kept small, it hardly ever runs.
template <int DP, int RED>
__device__ __forceinline__ float rescore(const unsigned char* row, const float* qs, int g) {
    float best = -INFINITY;
    const int n = RED == TB_GROUP_MAX ? g : 1, per = RED == TB_GROUP_MAX ? 1 : g;   // scores of a row, queries summed for each
#pragma unroll 1
    for (int u = 0; u < n; ++u) {
        float acc = 0.f, other = 0.f;                  // this chunk's chain and the other one's
#pragma unroll 1
        for (int c = 0; c < DP / 8; ++c) {
            float f[8];
            Elem<__nv_bfloat16>::unpack16(__ldcg(reinterpret_cast<const uint4*>(row) + c), f);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float q = 0.f;
#pragma unroll 1
                for (int i = 0; i < per; ++i) q += qs[(u + i) * DP + c * 8 + e];
                acc = fmaf(q, f[e], acc);
            }
            const float t = acc;
            acc = other, other = t;
        }
        best = RED == TB_GROUP_MAX ? fmaxf(best, acc + other) : acc + other;
    }
    return best;
}

// f(j, elements j .. j + 3) for every four of a thread's quarter of a query, of each of the g queries in head order.  `quarter` may
// be the caller's memory: 16 bytes at a time where that is aligned (`wide`), else 4.  (Staged in shared memory first, behind a
// barrier, the eight selections of a decode step over 32768 tokens take 7.5 us longer.)
template <int DP, typename F>
__device__ __forceinline__ void each_piece(const float* quarter, int g, bool wide, F&& f) {
    if (wide) {
#pragma unroll 4
        for (int u = 0; u < g; ++u)
#pragma unroll
            for (int j = 0; j < DP / 4; j += 4) f(j, *reinterpret_cast<const float4*>(quarter + u * DP + j));
    } else {
#pragma unroll 1
        for (int u = 0; u < g; ++u)
#pragma unroll
            for (int j = 0; j < DP / 4; j += 4) {
                const float* p = quarter + u * DP + j;
                f(j, make_float4(p[0], p[1], p[2], p[3]));
            }
    }
}

template <int DP, int RED>
struct FragScorer {
    static constexpr int kSteps = DP / 16, kTerms = 3, kRowBytes = DP * 2;
    typedef typename std::conditional<DP == 32, uint4, uint2>::type Piece;    // a thread's quarter of a row
    uint2 b[RED == TB_GROUP_SUM ? kSteps : 1];         // this lane's B fragments, per step
    const uint2* frag;                                 // ... or where they are in shared memory, [term][step][lane]
    // The largest bf16 term of (x, y), taken off them.  (The first one: a finite value does not become an infinity, above the
    // largest bf16 it takes that one.)
    __device__ __forceinline__ static uint32_t split(float& x, float& y, bool first = false) {
        const float top = 3.38953139e38f;
        const __nv_bfloat162 v = first ? __floats2bfloat162_rn(is_finite(x) ? fminf(fmaxf(x, -top), top) : x, is_finite(y) ? fminf(fmaxf(y, -top), top) : y)
                                       : __floats2bfloat162_rn(x, y);
        x -= __low2float(v), y -= __high2float(v);
        return *reinterpret_cast<const uint32_t*>(&v);
    }
    // Called by all threads of the block.  TB_GROUP_SUM: `qs` in shared or global memory, `wide` if 16-byte aligned;
    // TB_GROUP_MAX: staged and visible, `frags` holds kQueryFrags entries, one barrier.
    __device__ __forceinline__ void load_staged(const float* qs, int g, uint2* frags, bool wide = true) {
        const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
        // dimensions of word 2 st + half of the piece: tig * (DP / 4) + st * 4 + half * 2
        if constexpr (RED == TB_GROUP_SUM) {
            float x[kSteps * 2], y[kSteps * 2];
#pragma unroll
            for (int i = 0; i < kSteps * 2; ++i) x[i] = y[i] = 0.f;
            each_piece<DP>(qs + tig * (DP / 4), g, wide, [&](int j, float4 v) {
                x[j / 2] += v.x, y[j / 2] += v.y, x[j / 2 + 1] += v.z, y[j / 2 + 1] += v.w;
            });
#pragma unroll
            for (int i = 0; i < kSteps * 2; ++i) {
                const uint32_t high = split(x[i], y[i], true), middle = split(x[i], y[i]), low = split(x[i], y[i]);
                const uint32_t mine = (gid & 3) == 0 ? high : (gid & 3) == 1 ? middle : (gid & 3) == 2 ? low : 0u;
                if (i & 1) b[i >> 1].y = mine;
                else b[i >> 1].x = mine;
            }
        } else {
            const int st = threadIdx.x >> 5;
            frag = frags + lane;
            if (st < kSteps) {
                uint32_t t[kTerms][2];
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float2 v = *reinterpret_cast<const float2*>(qs + min(gid, g - 1) * DP + tig * (DP / 4) + st * 4 + half * 2);
#pragma unroll
                    for (int i = 0; i < kTerms; ++i) t[i][half] = split(v.x, v.y, i == 0);
                }
#pragma unroll
                for (int i = 0; i < kTerms; ++i) frags[(i * kSteps + st) * 32 + lane] = make_uint2(t[i][0], t[i][1]);
            }
            __syncthreads();
        }
    }
    // v[m]: this thread's piece of row 8 m + gid of the 32; d[m][2 i + e]: row 16 m + 8 i + gid, column 2 tig + e
    __device__ __forceinline__ void columns(const Piece (&v)[4], float (&d)[2][4]) const {
#pragma unroll
        for (int m = 0; m < 2; ++m) d[m][0] = d[m][1] = d[m][2] = d[m][3] = 0.f;
#pragma unroll
        for (int t = kTerms - 1; t >= 0; --t) {
            const uint2 b0 = frag[t * kSteps * 32];
            mma_16816(d[0], v[0].x, v[1].x, v[0].y, v[1].y, b0.x, b0.y);
            mma_16816(d[1], v[2].x, v[3].x, v[2].y, v[3].y, b0.x, b0.y);
            if constexpr (DP == 32) {
                const uint2 b1 = frag[(t * kSteps + 1) * 32];
                mma_16816(d[0], v[0].z, v[1].z, v[0].w, v[1].w, b1.x, b1.y);
                mma_16816(d[1], v[2].z, v[3].z, v[2].w, v[3].w, b1.x, b1.y);
            }
        }
    }
    // returns the score of the row this lane looks after (my_row)
    __device__ __forceinline__ float score(const Piece (&v)[4], int row0, int& my_row) const {
        const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
        // lane (gid, tig) takes row gid + 8 tig: accumulator pair 0 / 1 of the first 16 rows, then of the second
        my_row = row0 + gid + 8 * tig;
        float d[2][4], r[4];
        if constexpr (RED == TB_GROUP_SUM) {
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                d[m][0] = d[m][1] = d[m][2] = d[m][3] = 0.f;
                mma_16816(d[m], v[2 * m].x, v[2 * m + 1].x, v[2 * m].y, v[2 * m + 1].y, b[0].x, b[0].y);
                if constexpr (DP == 32) mma_16816(d[m], v[2 * m].z, v[2 * m + 1].z, v[2 * m].w, v[2 * m + 1].w, b[kSteps - 1].x, b[kSteps - 1].y);
                r[2 * m] = d[m][0] + d[m][1], r[2 * m + 1] = d[m][2] + d[m][3];
            }
        } else {
            columns(v, d);
            r[0] = fmaxf(d[0][0], d[0][1]), r[1] = fmaxf(d[0][2], d[0][3]), r[2] = fmaxf(d[1][0], d[1][1]), r[3] = fmaxf(d[1][2], d[1][3]);
#pragma unroll
            for (int i = 0; i < 4; ++i) r[i] = fmaxf(r[i], __shfl_xor_sync(0xffffffffu, r[i], 2));
        }
        const float lo = tig & 2 ? r[2] : r[0], hi = tig & 2 ? r[3] : r[1];
        const float mine = tig & 1 ? hi : lo, other = __shfl_xor_sync(0xffffffffu, tig & 1 ? lo : hi, 1);
        return RED == TB_GROUP_SUM ? mine + other : fmaxf(mine, other);
    }
    __device__ __forceinline__ static void load_piece(Piece& v, const unsigned char* quarter) { v = __ldcg(reinterpret_cast<const Piece*>(quarter)); }
};

// fp32 rows the same way: thread tig of a row's four takes a quarter of it, 32 rows per group, one FMA chain per quarter; three
// shuffles per four rows add the quarters and leave each lane the score of one row.  A row's score depends only on its bytes,
// and its sums are shorter than the two chains of row_score (rms error 2.1e-8 of sum |q k| for 2.5e-8).
template <int DP, int RED>
struct QuarterScorer {
    static constexpr int kRowBytes = DP * 4, kPer = DP / 16;                  // 16-byte pieces of a quarter
    struct Piece { uint4 w[kPer]; };
    float qr[RED == TB_GROUP_SUM ? DP / 4 : 1];
    const float* qs;
    int g;
    __device__ __forceinline__ void load_staged(const float* qs_, int g_, uint2*, bool wide = true) {
        const int tig = threadIdx.x & 3;
        qs = qs_ + tig * (DP / 4), g = g_;
        if constexpr (RED == TB_GROUP_SUM) {
#pragma unroll
            for (int j = 0; j < DP / 4; ++j) qr[j] = 0.f;
            each_piece<DP>(qs, g_, wide, [&](int j, float4 v) { qr[j] += v.x, qr[j + 1] += v.y, qr[j + 2] += v.z, qr[j + 3] += v.w; });
        }
    }
    __device__ __forceinline__ float reduce(const Piece (&v)[4], const float* q) const {
        const int tig = threadIdx.x & 3;
        float r[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            r[m] = 0.f;
#pragma unroll
            for (int c = 0; c < kPer; ++c) {
                float f[4];
                Elem<float>::unpack16(v[m].w[c], f);
#pragma unroll
                for (int e = 0; e < 4; ++e) r[m] = fmaf(q[c * 4 + e], f[e], r[m]);
            }
        }
        const float a0 = (tig & 2 ? r[2] : r[0]) + __shfl_xor_sync(0xffffffffu, tig & 2 ? r[0] : r[2], 2);
        const float a1 = (tig & 2 ? r[3] : r[1]) + __shfl_xor_sync(0xffffffffu, tig & 2 ? r[1] : r[3], 2);
        return (tig & 1 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, tig & 1 ? a0 : a1, 1);
    }
    __device__ __forceinline__ float score(const Piece (&v)[4], int row0, int& my_row) const {
        const int lane = threadIdx.x & 31;
        my_row = row0 + (lane >> 2) + 8 * (lane & 3);
        if constexpr (RED == TB_GROUP_SUM) return reduce(v, qr);
        float best = -INFINITY;
        for (int u = 0; u < g; ++u) best = fmaxf(best, reduce(v, qs + u * DP));
        return best;
    }
    __device__ __forceinline__ static void load_piece(Piece& v, const unsigned char* quarter) {
#pragma unroll
        for (int c = 0; c < kPer; ++c) v.w[c] = __ldcg(reinterpret_cast<const uint4*>(quarter) + c);
    }
};

// A group of 32 rows into a warp's registers: v[m] = this thread's quarter of row 8 m + gid; row(i) = address of row i < n.
template <typename Scorer, typename F>
__device__ __forceinline__ void load_rows(typename Scorer::Piece (&v)[4], int n, F&& row) {
    const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int m = 0; m < 4; ++m)
        if (8 * m + gid < n) Scorer::load_piece(v[m], row(8 * m + gid) + tig * (Scorer::kRowBytes / 4));
}

// The stream of a block of kW warps: rows [0, n) from `rows`, in groups of 32 dealt to the warps in turn, kU groups per warp in
// flight.  kWhole: n is a multiple of 32 (less code).  (Groups claimed from a counter as they are requested even out the warps, 1 us apart after 0.5 MB, but the claim is
// in every group's way: 32 problems of 32768 rows 20.1 -> 20.8 us.)
template <typename S, int kU, int kW, bool kWhole = false>
struct RowStream {
    typedef S Scorer;
    static constexpr int kGroupBytes = 32 * Scorer::kRowBytes;
    typename Scorer::Piece v[kU][4];
    const unsigned char* rows;
    int n, warp;
    __device__ __forceinline__ void load(int u, int g) {
        const unsigned char* first = rows + (size_t)g * kGroupBytes;
        if (kWhole ? g * 32 < n : g * 32 + 32 <= n) {  // warp-uniform
            const int lane = threadIdx.x & 31;
#pragma unroll
            for (int m = 0; m < 4; ++m) Scorer::load_piece(v[u][m], first + (8 * m + (lane >> 2)) * Scorer::kRowBytes + (lane & 3) * (Scorer::kRowBytes / 4));
        } else if (!kWhole && g * 32 < n) {            // the last one
            load_rows<Scorer>(v[u], n - g * 32, [&](int i) { return first + i * Scorer::kRowBytes; });
        }
    }
    // requests the groups [u0, u1) of every warp
    __device__ __forceinline__ void start(const unsigned char* rows_, int n_, int u0 = 0, int u1 = kU) {
        rows = rows_, n = n_, warp = threadIdx.x >> 5;
#pragma unroll
        for (int u = 0; u < kU; ++u)
            if (u >= u0 && u < u1) {
#pragma unroll
                for (int m = 0; m < 4; ++m) v[u][m] = {};
                load(u, u * kW + warp);
            }
    }
    // consume(slot, score) for every row
    template <typename F>
    __device__ __forceinline__ void run(const Scorer& scorer, F&& consume) {
        run_groups([&](const typename Scorer::Piece (&piece)[4], int row0) {
            int slot;
            const float sc = scorer.score(piece, row0, slot);
            return [=, &consume] { if (kWhole || slot < n) consume(slot, sc); };
        });
    }
    // f(slot) for every row that run() gives to this thread
    template <typename F>
    __device__ __forceinline__ void own_rows(F&& f) const {
        const int lane = threadIdx.x & 31;
#pragma unroll 1
        for (int slot = warp * 32 + (lane >> 2) + 8 * (lane & 3); slot < n; slot += kW * 32) f(slot);
    }
    // f(pieces, first row) for every group of 32; what it returns is called once the group's successor has been requested
    template <typename F>
    __device__ __forceinline__ void run_groups(F&& f) {
#pragma unroll 1
        for (int g0 = warp; g0 * 32 < n; g0 += kU * kW) {
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int g = g0 + u * kW;
                if (g * 32 >= n) break;                // warp-uniform
                auto rest = f(v[u], g * 32);
                load(u, g + kU * kW);
                rest();
            }
        }
    }
};

// Counts digits in a shared-memory histogram.  Nine keys in ten lie below a sampled bracket, in bin 0: added one by one to
// the same address they would cost a pass of the shared-memory pipe each (measured: 11 per instruction of 16 keys, half of
// a kernel's time), so that bin is counted in a register and added once, by flush().
struct DigitCounter {
    int below = 0;
    __device__ __forceinline__ void add(int* hist, int bin) {
        if (bin == 0) ++below;
        else asm volatile("red.shared.add.s32 [%0], 1;" ::"r"(smem_u32(hist + bin)) : "memory");
    }
    __device__ __forceinline__ void flush(int* hist) {   // whole warps; followed by a barrier
        below = warp_sum_int(below);
        if ((threadIdx.x & 31) == 0 && below) atomicAdd(hist, below);
        below = 0;
    }
};

// The same for keys that are mostly in the first or the last bin (a bin that is cut again): both are counted in a register, at
// most 65535 of each per thread.
template <int kLast>
struct EdgeCounter {
    uint32_t edges = 0;                                // below | above << 16
    __device__ __forceinline__ void add(int* hist, uint32_t bin) {
        if (bin - 1u < kLast - 1u) asm volatile("red.shared.add.s32 [%0], 1;" ::"r"(smem_u32(hist + bin)) : "memory");
        else edges += bin ? 0x10000u : 1u;
    }
    __device__ __forceinline__ void flush(int* hist) {   // whole warps; followed by a barrier
        const int below = warp_sum_int((int)(edges & 0xffffu)), above = warp_sum_int((int)(edges >> 16));
        if ((threadIdx.x & 31) == 0 && below) atomicAdd(hist, below);
        if ((threadIdx.x & 31) == 0 && above) atomicAdd(hist + kLast, above);
        edges = 0;
    }
};

// ---- from a bitmask of the candidates to the list -------------------------------------------------------
// Bit i of `mask` = candidate i (token lo + i) is selected; n_bits candidates, bits past them zero.

// Neighbour fetching on the mask (paper Sec. 3.4): `out` (as many words as mask, in other memory) = the selection with
// its neighbours, clipped to the candidates.  DILATE: every position within `radius`.  CLUSTER: every run of consecutive
// positions [a, b] gets radius * (b - a + 1) extra positions just outside, the larger half after b.  All threads call
// it, with `mask` complete and visible; `out` is visible to all on return.
template <int kThreads>
__device__ __forceinline__ void expand_mask(const uint32_t* mask, uint32_t* out, int n_bits, int radius, int nmode) {
    const int n_words = (n_bits + 31) / 32;
    const uint32_t last = n_bits & 31 ? (1u << (n_bits & 31)) - 1u : 0xffffffffu;
    if (nmode == TB_NEIGHBOR_DILATE) {
        for (int w = threadIdx.x; w < n_words; w += kThreads) {
            uint32_t m = mask[w];
            for (int d = 1; d <= radius; ++d) {        // bits d positions up and down
                const int wd = d >> 5, sh = d & 31;
                const uint32_t lo1 = w - wd >= 0 ? mask[w - wd] : 0u, lo2 = w - wd - 1 >= 0 ? mask[w - wd - 1] : 0u;
                const uint32_t hi1 = w + wd < n_words ? mask[w + wd] : 0u, hi2 = w + wd + 1 < n_words ? mask[w + wd + 1] : 0u;
                m |= __funnelshift_l(lo2, lo1, sh) | __funnelshift_r(hi1, hi2, sh);
            }
            out[w] = w == n_words - 1 ? m & last : m;
        }
        __syncthreads();
        return;
    }
    for (int w = threadIdx.x; w < n_words; w += kThreads) out[w] = mask[w];
    __syncthreads();
    auto mark = [&](long long from, long long to) {    // positions [from, to), clipped
        for (int x = (int)max(0ll, from); x < (int)min((long long)n_bits, to); ++x) atomicOr(&out[x >> 5], 1u << (x & 31));
    };
    for (int w = threadIdx.x; w < n_words; w += kThreads) {
        const uint32_t m = mask[w];
        uint32_t starts = m & ~((m << 1) | (w ? mask[w - 1] >> 31 : 0u));
        while (starts) {
            const int a = w * 32 + __ffs(starts) - 1;
            starts &= starts - 1;
            int e = a;                                 // first position behind the run
            while (e < n_words * 32) {
                const int sh = e & 31;
                const uint32_t rest = ~mask[e >> 5] >> sh;
                if (rest) { e += __ffs(rest) - 1; break; }
                e += 32 - sh;
            }
            e = min(e, n_bits);
            const long long n = (long long)radius * (e - a);
            mark(e, e + (n + 1) / 2), mark(a - n / 2, a);
        }
    }
    __syncthreads();
}

// Where a list goes: the context's (or the neighbour kernel's input), and the caller's copy.
struct ListOut {
    int32_t* idx;
    int32_t* cnt;
    int32_t* idx_copy;
    int32_t* cnt_copy;
    int radius, nmode, cap;
    __device__ __forceinline__ ListOut(const Geom& gm, const SelectArgs& a, size_t state_row, int launch_row, int32_t* state_idx, int32_t* state_cnt) {
        const size_t row = a.dst_is_state ? state_row : (size_t)launch_row;
        idx = (a.dst_is_state ? state_idx : a.idx_dst) + row * a.idx_stride;
        cnt = (a.dst_is_state ? state_cnt : a.cnt_dst) + row;
        idx_copy = a.idx_copy ? a.idx_copy + (size_t)launch_row * gm.idx_cap : nullptr;
        cnt_copy = a.cnt_copy ? a.cnt_copy + launch_row : nullptr;
        radius = a.radius, nmode = a.nmode, cap = a.idx_stride;
    }
    __device__ __forceinline__ void count(int n) const {   // one thread
        *cnt = n;
        if (cnt_copy) *cnt_copy = n;
    }
    // every candidate (neighbours add nothing), or none
    template <int kThreads>
    __device__ __forceinline__ void all(int lo, int n) const {
        for (int i = threadIdx.x; i < n; i += kThreads) {
            idx[i] = lo + i;
            if (idx_copy) idx_copy[i] = lo + i;
        }
        if (threadIdx.x == 0) count(max(n, 0));
    }
};

// Writes the ascending list of a mask: its first `limit` positions, as tokens, to dst and (unless null) to copy.
// Returns the number of bits.  A thread owns a run of 16-bit half words; `slots` holds kThreads / 32 ints.
template <int kThreads>
__device__ __forceinline__ int write_mask_list(const uint32_t* mask, int n_bits, int lo, int limit, int32_t* __restrict__ dst,
                                               int32_t* __restrict__ copy, int* slots) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint16_t* mask16 = reinterpret_cast<const uint16_t*>(mask);
    const int n_half = (n_bits + 15) / 16;
    const int per = (n_half + kThreads - 1) / kThreads;
    const int w0 = min(n_half, (int)threadIdx.x * per), w1 = min(n_half, w0 + per);
    int cnt = 0;
    for (int w = w0; w < w1; ++w) cnt += __popc((uint32_t)mask16[w]);
    const int incl = warp_incl_scan(cnt, lane);
    if (lane == 31) slots[warp] = incl;
    __syncthreads();
    int o = incl - cnt, total = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        const int x = slots[w];
        total += x;
        o += w < warp ? x : 0;
    }
    for (int w = w0; w < w1; ++w) {
        uint32_t bits = mask16[w];
        while (bits) {
            const int t = lo + w * 16 + __ffs(bits) - 1;
            bits &= bits - 1;
            if (o < limit) {
                dst[o] = t;
                if (copy) copy[o] = t;
            }
            ++o;
        }
    }
    return total;
}

// From the mask to the finished list; `other` = room for a second mask (radius > 0 only).  All threads, mask visible.
template <int kThreads>
__device__ __forceinline__ void finish_mask_list(const uint32_t* mask, uint32_t* other, int n_bits, int lo, const ListOut& out, int* slots) {
    if (out.radius > 0) {
        expand_mask<kThreads>(mask, other, n_bits, out.radius, out.nmode);
        mask = other;
    }
    const int total = write_mask_list<kThreads>(mask, n_bits, lo, out.cap, out.idx, out.idx_copy, slots);
    if (threadIdx.x == 0) out.count(total);
}

}  // namespace tb
