// Selection of long problems: scoring, exact top-B, neighbour fetching and the copy of the list for the caller, a cluster
// of blocks per (layer, sequence, list), one launch (paper Sec. 3.4, Sec. 4 "Token Selection Policy").
//
// What bounds it is the projected keys' way from HBM, so a block is built to stream: 512 threads, one block per SM, rows
// straight into tensor-core fragments (fp32: into the lanes that multiply them), 128 KB of them in flight, no shared memory,
// no barrier and no copy engine between a row and its score.  What stays on chip is a row's score or, where a block has too many
// rows for that, the two bytes of its first digit.
//   sample   the same 64 rows in every block of the cluster bracket where the B-th largest score will fall: equal slices of
//            score across the bracket, an open bin on either side.  The digit is monotone in the score whatever the sample
//            says: the result never depends on it, only how few rows share the threshold's bin does
//   stream   score, digit, histogram
//   cluster  every block sends its histogram (16-bit counts) to every peer, one cluster barrier; all find the same bin
//   finish   scores -> bitmask; the few rows inside the bin go to every peer's list (second barrier), each block ranks them
//            itself (equal keys by position) and writes its part of the ascending list from its part of the bitmask
//   neighbours (if asked for)  bitmasks to every peer (third barrier), each block expands all of it and writes its part
// A crowded bin (an outlier that stretches the bracket, a threshold outside of it, ties) is cut into slices again, now of the
// order-preserving 32-bit key, from the scores on chip or, where only the digits fit, from the rows, until it is small or one
// key wide: a few rounds at most, each a thousand times finer.
// Nothing waits for anything but cluster barriers and the block's own loads.
#include "tb_select.cuh"

namespace tb {

namespace {

constexpr int kSampleRows = 64;
constexpr int kMaxRank = 256;       // keys of the threshold bin that are ranked pairwise
constexpr int kMaxBlocks = 16;      // per cluster (more than 8: non-portable)
constexpr int kMaxShare = 65408;    // rows of a cluster's block: 16-bit counts, whole 128-row pieces
constexpr size_t kScoresSmem = 194 * 1024;   // loads in flight need room in L1: 48000 rows with their scores (221 KB) 75 us, without 62

// kThreads: 512, one block per SM, or 256, two; 128 registers per thread and 128 KB of rows in flight per SM either way.
template <int kThreads>
struct __align__(16) StreamSmem {
    static constexpr int kBins = 4 * kThreads, kWarps = kThreads / 32;
    int hist[kBins];
    uint2 cand[kMaxRank];           // (key, candidate) of the threshold bin, all blocks'
    uint2 mine[kMaxRank];           // (key, own row) of this block's
    float qs[kMaxGroup * 32];       // the list's importance queries
    uint2 frags[kQueryFrags];       // ... as tensor-core operands (TB_GROUP_MAX)
    uint32_t sample[kSampleRows];
    int slots[2][32];               // per warp; zero past kWarps
    // per block: keys in the threshold bin, those of the lower blocks, and those that are taken
    int inbin[kMaxBlocks], inbin_before[kMaxBlocks], winners[kMaxBlocks];
    uint32_t s_lo, s_hi;
    int bin, krem, count, n_mine, lower, total;
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_smem(const void* p, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void store_peer(uint32_t at, uint2 v) {
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(at), "r"(v.x), "r"(v.y) : "memory");
}

// 2 bits + (x >= y)
__device__ __forceinline__ uint32_t push_ge(uint32_t bits, uint32_t x, uint32_t y) {
    uint32_t r;
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %2;\n\taddc.u32 %0, %3, %3;\n\t}" : "=r"(r) : "r"(x), "r"(y), "r"(bits));
    return r;
}

// NaN stays: what is not a number goes to the lowest bin and takes no number's place.
__device__ __forceinline__ float min_or_nan(float x, float y) {
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(x), "f"(y));
    return r;
}

__device__ __forceinline__ float key_score(uint32_t key) { return __uint_as_float(key & 0x80000000u ? key & 0x7fffffffu : ~key); }

// Bins, monotone in the score: equal slices of score or, once one of these was too full, slices of 2^shift keys from base up; the
// first one also holds everything below, the last one everything above.
template <int kBins>
struct Slices {
    float scale, off;               // slices of score (shift < 0): score * scale + off
    uint32_t base;                  // slices of keys
    int shift;
    __device__ __forceinline__ bool linear() const { return shift < 0; }
    __device__ __forceinline__ float place(float score) const { return min_or_nan(fmaf(score, scale, off), (float)(kBins - 1)); }
    __device__ __forceinline__ uint32_t linear_bin(float score) const { return __float2uint_rz(place(score)); }   // (below 0, and NaN, becomes 0)
    __device__ __forceinline__ uint32_t key_bin(uint32_t key) const { return min((max(key, base) - base) >> shift, (uint32_t)(kBins - 1)); }
    __device__ __forceinline__ uint32_t bin(float score) const { return linear() ? linear_bin(score) : key_bin(order_key(score)); }
    // from the keys of the sample scores that bracket the threshold; `reach` times as far up as they are apart, since of 64 rows
    // none may be in the upper 2 %
    __device__ __forceinline__ void bracket(uint32_t s_lo, uint32_t s_hi, float reach) {
        const float lo = key_score(s_lo), width = key_score(s_hi) - lo;
        scale = (float)(kBins - 2) / (reach * width), off = 1.f - lo * scale;
        if (!(scale > 0.f && is_finite(scale) && is_finite(off))) scale = 1.f, off = 0.f;   // equal, infinite: any slices will do
        shift = -1;
    }
    // the finest slices that cover the keys from .. last with neither the first nor the last of them (unless from is near 0)
    __device__ __forceinline__ void cover(uint32_t from, uint32_t last) {
        const uint32_t range = last - from;
        shift = max(0, 1 + __clz(kBins) - __clz(range));
        if ((range >> shift) > (uint32_t)(kBins - 3)) ++shift;
        base = from - min(from, 1u << shift);
    }
    __device__ __forceinline__ bool one_key(int b) const { return shift == 0 && b < kBins - 1 && (b > 0 || base == 0u); }
    // Finer slices for bin b (not one_key).  Above or below the bracket: first twice the bracket, further on, which is where the
    // threshold will be.  A slice of score ends at about these keys; should the threshold be beyond, the next cut finds it in the
    // open bin there.
    __device__ __forceinline__ void cut(int b) {
        const float next = b == 0 ? off * 0.5f + (float)(kBins - 2) : off * 0.5f - (float)(kBins - 4) * 0.5f;
        if (shift == -1 && (b == 0 || b == kBins - 1) && is_finite(next)) {
            scale *= 0.5f, off = next, shift = -2;
            return;
        }
        uint32_t from = base + ((uint32_t)b << (shift & 31)), last = from + ((1u << (shift & 31)) - 1u);
        if (linear()) from = order_key(((float)b - 0.01f - off) / scale), last = max(from, order_key(((float)b + 1.01f - off) / scale));
        cover(b == 0 ? 0u : from, b == kBins - 1 ? 0xffffffffu : last);
    }
};

// Exclusive prefix of `v` over the block in thread order, and the block's total.  One barrier; `slots` (32 ints, zero past
// the block's warps) must not be written again before the next one.
__device__ __forceinline__ int block_excl_scan(int v, int* slots, int& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int incl = warp_incl_scan(v, lane);
    if (lane == 31) slots[warp] = incl;
    __syncthreads();
    const int w = slots[lane], upto = warp_incl_scan(w, lane);
    total = __shfl_sync(0xffffffffu, upto, 31);
    return __shfl_sync(0xffffffffu, upto - w, warp) + incl - v;
}

// The bin that holds the k-th largest of the counted keys (thread t holds the counts of bins 4 t .. 4 t + 3): all threads get
// it, with k' = k - keys in higher bins and the bin's population.  1 <= k <= total.
template <typename Smem>
__device__ __forceinline__ void find_bin(Smem* sm, const int (&b)[4], int k, int& bin, int& krem, int& count) {
    const int tid = threadIdx.x, mine = (b[0] + b[1]) + (b[2] + b[3]);
    int total;
    const int below = block_excl_scan(mine, sm->slots[0], total);
    int run = total - below - mine;                    // keys in bins above this thread's
    if (run < k && k <= run + mine) {                  // exactly one thread
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            if (run < k && k <= run + b[i]) sm->bin = tid * 4 + i, sm->krem = k - run, sm->count = b[i];
            run += b[i];
        }
    }
    __syncthreads();
    bin = sm->bin, krem = sm->krem, count = sm->count;
}

// Writes the tokens of mask words [w0, w1) in ascending order: list entries base, base + 1, ...
template <int kThreads>
__device__ __forceinline__ void write_words(StreamSmem<kThreads>* sm, const uint32_t* mask, int w0, int w1, int base, int lo, const ListOut& out) {
    const uint16_t* mask16 = reinterpret_cast<const uint16_t*>(mask);
    const int n_half = 2 * (w1 - w0), per = (n_half + kThreads - 1) / kThreads;
    const int h0 = 2 * w0 + min(n_half, (int)threadIdx.x * per), h1 = min(2 * w1, h0 + per);
    int cnt = 0, total;
    for (int h = h0; h < h1; ++h) cnt += __popc((uint32_t)mask16[h]);
    int o = base + block_excl_scan(cnt, sm->slots[1], total);
    for (int h = h0; h < h1; ++h) {
        uint32_t bits = mask16[h];
        while (bits) {
            const int t = lo + h * 16 + __ffs(bits) - 1;
            bits &= bits - 1;
            if (o < out.cap) {
                out.idx[o] = t;
                if (out.idx_copy) out.idx_copy[o] = t;
            }
            ++o;
        }
    }
}

// The (layer, sequence) pairs of a launch, longest first: layer << 8 | sequence.
struct StreamOrder {
    uint16_t pair[kMaxLaunchUnits];
};

template <typename T, int DP, int RED, int kThreads>
struct StreamTypes {
    static constexpr bool kMma = Elem<T>::kBytes == 2;
    typedef typename std::conditional<kMma, FragScorer<DP, RED>, QuarterScorer<DP, RED>>::type Scorer;
    static constexpr int kU = kMma && DP == 16 ? 8 : !kMma && DP == 32 ? 2 : 4;   // 8 KB in flight per warp
    typedef RowStream<Scorer, kU, kThreads / 32, true> Stream;
};

template <typename T, int DP, int RED, int kThreads>
__global__ void __launch_bounds__(kThreads, 512 / kThreads) select_stream_kernel(const unsigned char* __restrict__ kimp, Geom gm, UnitTable ut, StreamOrder order,
                                                                                 SelectArgs a, int room, int most, int keep_scores, int32_t* __restrict__ state_idx,
                                                                                 int32_t* __restrict__ state_cnt, int32_t* __restrict__ status) {
    typedef StreamTypes<T, DP, RED, kThreads> Types;
    typedef StreamSmem<kThreads> Smem;
    typedef typename Types::Scorer Scorer;
    constexpr int kBins = Smem::kBins, kWarps = Smem::kWarps;
    constexpr bool kMma = Types::kMma;
    constexpr int RB = Scorer::kRowBytes;
    uint32_t C_, rank_;
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C_));
    asm volatile("mov.u32 %0, %%cluster_ctaid.x;" : "=r"(rank_));
    const int C = (int)C_, rank = (int)rank_;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem* sm = reinterpret_cast<Smem*>(smem_raw);
    uint16_t* peer_hist = reinterpret_cast<uint16_t*>(sm + 1);                    // [C][kBins] (C > 1)
    const int mask_words = (a.radius > 0 ? C * room : room) / 32;
    uint32_t* mask = reinterpret_cast<uint32_t*>(peer_hist + (C > 1 ? C * kBins : 0));   // the block's part, or (neighbours) the problem's
    uint32_t* wider = mask + mask_words;                                          // neighbours only
    float* scores = reinterpret_cast<float*>(wider + (a.radius > 0 ? mask_words : 0));   // [room], keep_scores,
    uint16_t* digits = reinterpret_cast<uint16_t*>(scores);                       // or [room]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const int ll = order.pair[blockIdx.z] >> 8, s = order.pair[blockIdx.z] & 0xff, h = blockIdx.y, unit = (ll * ut.n_seq + s) * gm.Hl + h;
    const size_t cu = list_unit(gm, ut, ll, s, h);
    const ListOut out(gm, a, cu, unit, state_idx, state_cnt);
    reinterpret_cast<int4*>(sm->hist)[tid] = make_int4(0, 0, 0, 0);
    if (tid < 64) sm->slots[0][tid] = 0;
    if (tid == 0) sm->n_mine = sm->lower = sm->total = 0;
    const int L = unit_len(gm, ut, ll, s);
    const int lo = min(a.sinks, L), hi = max(lo, L - a.recent);
    const int ncand = candidates_within(hi - lo, most, status), k = min(a.budget, ncand);
    check_candidates_projected(gm, ut, ll, s, hi, status);
    if (k <= 0 || k == ncand) {                        // nothing to rank (uniform over the cluster): none, or all (neighbours add nothing then)
        for (int i = rank * kThreads + tid; i < k; i += C * kThreads) {
            out.idx[i] = lo + i;
            if (out.idx_copy) out.idx_copy[i] = lo + i;
        }
        if (rank == 0 && tid == 0) out.count(max(k, 0));
        return;
    }
    // this block's rows: candidates slot0 .. slot0 + n_local - 1, whole words of the bitmask
    const int share = min(room, ((ncand + C - 1) / C + 127) & ~127);
    const int slot0 = min(ncand, rank * share), n_local = min(share, ncand - slot0);
    const unsigned char* stream = kimp + ((size_t)key_unit(gm, ut, ll, s, h) * gm.max_seq_len + lo) * RB;
    const unsigned char* rows = stream + (size_t)slot0 * RB;

    // ---- what is waited for first is requested first: the queries, the sample, one group of rows per warp ---------------
    // (With all of the opening rows requested at once the sample queues behind the other warps' and blocks'.)
    const float* q_unit = a.q_imp + query_row(gm, ut, ll, s, h) * DP;
    const float q_elem = tid < gm.gl * DP ? __ldg(q_unit + tid) : 0.f;            // (staged where every lane wants all of it, and for rescore)
    typename Scorer::Piece few[4];                     // warps 0 and 1: 32 sample rows each; warp 2: the rows past the last whole group
    const int n_whole = n_local & ~31, n_tail = warp == kSampleRows / 32 ? n_local - n_whole : 0;
    if (warp <= kSampleRows / 32)
        load_rows<Scorer>(few, warp < kSampleRows / 32 ? 32 : n_tail, [&](int i) {
            return warp < kSampleRows / 32 ? stream + (size_t)((long long)(warp * 32 + i) * ncand / kSampleRows) * RB : rows + (size_t)(n_whole + i) * RB;
        });
    typename Types::Stream rs;
    rs.start(rows, n_whole, 0, 1);
    if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // (waited for before the first remote store)
    if (tid < gm.gl * DP) sm->qs[tid] = q_elem;
    Scorer scorer;
    bool odd_query = false;                            // (a summed query that is not finite shows in every score)
    if constexpr (RED == TB_GROUP_SUM) {
        scorer.load_staged(q_unit, gm.gl, nullptr, (reinterpret_cast<uintptr_t>(a.q_imp) & 15u) == 0u);   // (queries start at any float)
    } else {
        odd_query = __syncthreads_or(kMma && !is_finite(q_elem));
        scorer.load_staged(sm->qs, gm.gl, sm->frags);
    }

    // about p * kSampleRows sample keys lie above the threshold (p = k / candidates): +- 4 standard deviations of that rank, one
    // more down and a longer reach up where a second look costs the rows again (eight 64K
    // sequences, a step of four layers: 261 us, 348 with the narrow bracket)
    const float p = (float)k / (float)ncand, mean = p * kSampleRows, sd = sqrtf(mean * (1.f - p));
    const int r_hi = max(0, (int)floorf(mean - 4.f * sd) - 1), r_lo = min(kSampleRows - 1, (int)ceilf(mean + (keep_scores ? 4.f : 5.f) * sd) + 1);
    Slices<kBins> sl;
    if (warp < kSampleRows / 32) {
        int at;
        const float sc = scorer.score(few, warp * 32, at);
        sm->sample[at] = order_key(sc);
    }
    rs.start(rows, n_whole, 1, Types::kU);
    __syncthreads();
    {                                                  // descending ranks (equal keys by index), some keys per warp
        const uint32_t x0 = sm->sample[lane], x1 = sm->sample[lane + 32];
#pragma unroll
        for (int i = 0; i < kSampleRows / kWarps; ++i) {
            const int at = warp * (kSampleRows / kWarps) + i;
            const uint32_t me = sm->sample[at];
            const int r = __popc(__ballot_sync(0xffffffffu, x0 > me || (x0 == me && lane < at))) +
                          __popc(__ballot_sync(0xffffffffu, x1 > me || (x1 == me && lane + 32 < at)));
            if (lane == 0 && r == r_hi) sm->s_hi = me;
            if (lane == 0 && r == r_lo) sm->s_lo = me;
        }
    }
    __syncthreads();
    sl.bracket(sm->s_lo, sm->s_hi, !keep_scores ? 6.f : mean < 3.f ? 4.5f : 3.f);

    // ---- rounds: one, hardly ever more ---------------------------------------------------------------------------------
    DigitCounter counter;
    int bin, kr, bc;
    bool whole, ties = false;
#pragma unroll 1
    for (bool first = true;; first = false) {
        auto put = [&](int slot, float score, uint32_t d) {
            if (keep_scores) scores[slot] = score;
            else digits[slot] = (uint16_t)d;
            return (int)d;
        };
        bool odd = false;
        if (first) {
            float sum = 0.f;
            auto consume = [&](int slot, float sc) {
                sum += sc;
                counter.add(sm->hist, put(slot, sc, sl.linear_bin(sc)));
            };
            if (n_tail) {
                int slot;
                const float sc = scorer.score(few, n_whole, slot);
                if (slot < n_local) consume(slot, sc);
            }
            rs.run(scorer, consume);
            odd = kMma && (odd_query || !is_finite(sum));
        } else {
            EdgeCounter<kBins - 1> recount;            // (nearly all rows are below or above the slices by now)
            if (keep_scores) {
                for (int i = tid; i < n_local; i += kThreads) recount.add(sm->hist, sl.bin(scores[i]));
            } else {
                // Rows outside the bin stay above or below it: only a group of 32 with one inside is read again.  256 lists of 65536 of
                // which a few per launch have 250 or 350 equal keys at their threshold: 242 and 304 us, with all rows read again 288
                // and 367, without such lists 197.  (Not scoring the other groups either: 222 and 260, but the code is in the way of
                // launches that never come here, 337.5 -> 339.8 us per decode step at 32K.)
#pragma unroll 1
                for (int g0 = warp * 32; g0 < n_local; g0 += kThreads) {
                    if (__any_sync(0xffffffffu, g0 + lane < n_local && digits[g0 + lane] == bin))
                        load_rows<Scorer>(few, n_local - g0, [&](int i) { return rows + (size_t)(g0 + i) * RB; });
                    int slot;
                    const float sc = scorer.score(few, g0, slot);   // (of rows that are not there, or of others: not used)
                    if (slot < n_local) {
                        const int d = digits[slot];
                        recount.add(sm->hist, put(slot, sc, d == bin ? sl.bin(sc) : d > bin ? kBins - 1 : 0));
                        if (kMma) odd = odd || (d == bin && (odd_query || !is_finite(sc)));
                    }
                }
            }
            __syncwarp();
            recount.flush(sm->hist);
        }
        counter.flush(sm->hist);
        if (__syncthreads_or(odd)) {                   // infinite scores, or scores dropped beside an infinite query (see FragScorer)
            if constexpr (kMma)
                for (int i = tid; i < n_local; i += kThreads) {
                    const float sc = rescore<DP, RED>(rows + (size_t)i * RB, sm->qs, gm.gl);
                    if (is_finite(sc)) continue;
                    atomicAdd(&sm->hist[keep_scores ? sl.bin(scores[i]) : (uint32_t)digits[i]], -1);
                    atomicAdd(&sm->hist[put(i, sc, sl.bin(sc))], 1);
                }
            __syncthreads();
        }

        // ---- threshold bin, from every block's histogram ---------------------------------------------------------------
        int b[4];
        {
            const int4 x = reinterpret_cast<const int4*>(sm->hist)[tid];
            b[0] = x.x, b[1] = x.y, b[2] = x.z, b[3] = x.w;
        }
        int low[4] = {0, 0, 0, 0};                     // in the lower blocks
        if (C > 1) {
            const uint2 packed = make_uint2((uint32_t)b[0] | (uint32_t)b[1] << 16, (uint32_t)b[2] | (uint32_t)b[3] << 16);
            if (first) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every peer runs
            const uint2* mine = reinterpret_cast<const uint2*>(peer_hist + rank * kBins) + tid;
            for (int r = 0; r < C; ++r) store_peer(peer_smem(mine, rank + r < C ? rank + r : rank + r - C), packed);
            cluster_sync();
            b[0] = b[1] = b[2] = b[3] = 0;
            for (int r = 0; r < C; ++r) {
                const uint2 x = reinterpret_cast<const uint2*>(peer_hist + r * kBins)[tid];
                const int c0 = (int)(x.x & 0xffffu), c1 = (int)(x.x >> 16), c2 = (int)(x.y & 0xffffu), c3 = (int)(x.y >> 16);
                b[0] += c0, b[1] += c1, b[2] += c2, b[3] += c3;
                if (r < rank) low[0] += c0, low[1] += c1, low[2] += c2, low[3] += c3;
            }
        }
        find_bin(sm, b, k, bin, kr, bc);
        whole = bc == kr;
        ties = !whole && bc > kMaxRank && sl.one_key(bin);
        if (whole || ties || bc <= kMaxRank) {
            int la = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) la += tid * 4 + i > bin ? low[i] : 0;
            la = warp_sum_int(la);
            if (lane == 0 && la) atomicAdd(&sm->lower, la);
            if (warp == kWarps - 1) {
                const int n = lane >= C ? 0 : C > 1 ? (int)peer_hist[lane * kBins + bin] : bc, before = warp_incl_scan(n, lane) - n;
                if (lane < C) sm->inbin[lane] = n, sm->inbin_before[lane] = before, sm->winners[lane] = whole ? n : ties ? max(0, min(n, kr - before)) : 0;
            }
            break;
        }
        sl.cut(bin);
        reinterpret_cast<int4*>(sm->hist)[tid] = make_int4(0, 0, 0, 0);
        if (C > 1) cluster_sync(); else __syncthreads();   // the histograms have been read
    }

    // ---- scores or digits -> bitmask ------------------------------------------------------------------------------------------
    const int word0 = a.radius > 0 ? slot0 / 32 : 0, n_words = (n_local + 31) / 32;
    {
        uint8_t* mask8 = reinterpret_cast<uint8_t*>(mask + word0);
        // What is compared: digits, places among the slices of score (positive floats are ordered like their bits), or keys; the
        // first that belongs to the bin, and the first above it, which may not exist.  A verdict is a carry.
        const bool place = keep_scores && sl.linear(), by_key = keep_scores && !sl.linear();
        const uint64_t end = (uint64_t)sl.base + ((uint64_t)(bin + 1) << (by_key ? sl.shift : 0));
        const uint32_t from = place ? __float_as_uint((float)bin) : !by_key ? (uint32_t)bin : bin == 0 ? 0u : sl.base + ((uint32_t)bin << sl.shift);
        const uint32_t above = whole ? from : place ? __float_as_uint((float)(bin + 1)) : !by_key ? (uint32_t)bin + 1u : (uint32_t)end;
        const bool none_above = !whole && (bin == kBins - 1 || (by_key && end > 0xffffffffull));
        for (int v = tid; v < (n_local + 127) / 128 * 16; v += kThreads) {
            uint32_t d[8];
            if (keep_scores) {
                const float4 x = reinterpret_cast<const float4*>(scores)[2 * v], y = reinterpret_cast<const float4*>(scores)[2 * v + 1];
                const float f[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) d[e] = place ? __float_as_uint(fmaxf(sl.place(f[e]), 0.f)) : order_key(f[e]);
            } else {
                const uint4 x = reinterpret_cast<const uint4*>(digits)[v];
                d[0] = x.x & 0xffffu, d[1] = x.x >> 16, d[2] = x.y & 0xffffu, d[3] = x.y >> 16;
                d[4] = x.z & 0xffffu, d[5] = x.z >> 16, d[6] = x.w & 0xffffu, d[7] = x.w >> 16;
            }
            uint32_t take = 0u, in = 0u;
#pragma unroll
            for (int e = 7; e >= 0; --e) take = push_ge(take, d[e], above), in = push_ge(in, d[e], from);
            take = none_above ? 0u : take, in &= ~take;
            const int left = n_local - v * 8;
            const uint32_t valid = left >= 8 ? 0xffu : left > 0 ? (1u << left) - 1u : 0u;
            mask8[v] = (uint8_t)(take & valid);
            in = whole || ties ? 0u : in & valid;
            while (in) {                               // rare: a handful of rows per block
                const int row = v * 8 + __ffs(in) - 1;
                in &= in - 1;
                sm->mine[atomicAdd(&sm->n_mine, 1)] = make_uint2(keep_scores ? order_key(scores[row]) : 0u, (uint32_t)row);
            }
        }
    }
    __syncthreads();
    if (ties) {
        // equal keys: the first ones in position order are taken; a thread owns a run of words
        const int per = (n_words + kThreads - 1) / kThreads, w0 = min(n_words, tid * per), w1 = min(n_words, w0 + per);
        auto equals = [&](int w) {
            uint32_t eq = 0u;
            for (int i = w * 32; i < min(n_local, w * 32 + 32); ++i)
                eq |= (uint32_t)((keep_scores ? sl.bin(scores[i]) : (uint32_t)digits[i]) == (uint32_t)bin) << (i & 31);
            return eq;
        };
        int n_eq = 0, total;
        for (int w = w0; w < w1; ++w) n_eq += __popc(equals(w));
        int before = block_excl_scan(n_eq, sm->slots[0], total);
        for (int w = w0; w < w1; ++w) {
            uint32_t eq = equals(w), take = 0u;
            while (eq && before < sm->winners[rank]) take |= eq & (0u - eq), eq &= eq - 1, ++before;
            mask[word0 + w] |= take;
        }
        __syncthreads();
    } else if (!whole) {
        // this block's rows inside the bin: their keys, then all of them to every block
        const int n_mine = sm->n_mine;                 // <= bc <= kMaxRank
        const int cand_base = sm->inbin_before[rank];
        if (!keep_scores) {                              // (the rows again, and their scores)
            for (int e0 = warp * 32; e0 < n_mine; e0 += kThreads) {
                load_rows<Scorer>(few, n_mine - e0, [&](int i) { return rows + (size_t)sm->mine[e0 + i].y * RB; });
                int e;
                float sc = scorer.score(few, e0, e);
                if (e < n_mine) {
                    if constexpr (kMma)
                        if (odd_query || !is_finite(sc)) sc = rescore<DP, RED>(rows + (size_t)sm->mine[e].y * RB, sm->qs, gm.gl);
                    sm->mine[e].x = order_key(sc);
                }
            }
            __syncthreads();
        }
        if ((tid & (kMaxBlocks - 1)) < C)
            for (int e = tid / kMaxBlocks; e < n_mine; e += kThreads / kMaxBlocks)
                store_peer(peer_smem(&sm->cand[cand_base + e], tid & (kMaxBlocks - 1)), make_uint2(sm->mine[e].x, sm->mine[e].y + (uint32_t)slot0));
        if (C > 1) cluster_sync(); else __syncthreads();
        // rank: larger key first, equal keys by position; eight lanes per entry
        for (int e0 = 0; e0 < bc; e0 += kThreads / 8) {
            const int e = e0 + tid / 8;
            const uint2 it = sm->cand[min(e, bc - 1)];
            int before = 0;
            for (int j = tid & 7; j < bc; j += 8) {
                const uint2 o = sm->cand[j];
                before += (o.x > it.x) | ((o.x == it.x) & (o.y < it.y));
            }
#pragma unroll
            for (int off = 1; off < 8; off <<= 1) before += __shfl_xor_sync(0xffffffffu, before, off);
            if ((tid & 7) == 0 && e < bc && before < kr) {
                int r_of = C - 1;
                while (e < sm->inbin_before[r_of]) --r_of;
                atomicAdd(&sm->winners[r_of], 1);
                if (r_of == rank) {
                    const int ls = (int)it.y - slot0;
                    atomicOr(&mask[word0 + (ls >> 5)], 1u << (ls & 31));
                }
            }
        }
        __syncthreads();
    }
    pdl_launch_dependents();                           // what is left is short; a successor waits for this grid's completion

    // ---- neighbours and list ------------------------------------------------------------------------------------------------
    if (a.radius == 0) {
        int base = sm->lower;
        for (int r = 0; r < rank; ++r) base += sm->winners[r];
        write_words(sm, mask, 0, n_words, base, lo + slot0, out);
        if (rank == 0 && tid == 0) out.count(k);
        return;
    }
    if (C > 1) {
        const int n16 = (n_local + 127) / 128;         // 16-byte pieces of this block's words
        for (int t = tid; t < n16 * (C - 1); t += kThreads) {
            const int v = t / (C - 1), r = t - v * (C - 1);
            const uint4 x = reinterpret_cast<const uint4*>(mask + word0)[v];
            asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(peer_smem(mask + word0 + v * 4, r < rank ? r : r + 1)), "r"(x.x), "r"(x.y),
                         "r"(x.z), "r"(x.w)
                         : "memory");
        }
        cluster_sync();
    }
    expand_mask<kThreads>(mask, wider, ncand, a.radius, a.nmode);
    int before = 0, total = 0;
    for (int w = tid; w < (ncand + 31) / 32; w += kThreads) {
        const int n = __popc(wider[w]);
        total += n, before += w < word0 ? n : 0;
    }
    total = warp_sum_int(total), before = warp_sum_int(before);
    if (lane == 0) atomicAdd(&sm->total, total), sm->slots[0][warp] = before;
    __syncthreads();
    before = warp_sum_int(sm->slots[0][lane]);
    write_words(sm, wider, word0, word0 + n_words, before, lo, out);
    if (rank == 0 && tid == 0) out.count(sm->total);
}

size_t stream_smem(int threads, int C, int room, bool neighbours, bool scores) {
    return (threads == 512 ? sizeof(StreamSmem<512>) : sizeof(StreamSmem<256>)) + (C > 1 ? (size_t)C * threads * 8 : 0) +
           (neighbours ? 2 * (size_t)C : 1) * (room / 8) + (size_t)room * (scores ? 4 : 2);
}

struct StreamLaunch {
    cudaLaunchConfig_t cfg;
    int room, most, keep_scores;    // rows of a block, candidates of a problem, scores (and not digits) on chip
    int* fit;                       // only asks how many clusters run at once
};

template <typename T, int DP, int RED, int kThreads>
cudaError_t launch(const tb_ctx* c, const UnitTable& ut, const StreamOrder& order, const SelectArgs& a, const StreamLaunch& l) {
    const auto kernel = select_stream_kernel<T, DP, RED, kThreads>;
    static DeviceFlags done;
    const cudaError_t configured = once_per_device(done, [&] {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        if (e != cudaSuccess) return e;
        (void)cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        (void)cudaGetLastError();
        return e;
    });
    if (configured != cudaSuccess) return configured;
    if (l.fit) {
        if (cudaOccupancyMaxActiveClusters(l.fit, kernel, &l.cfg) != cudaSuccess) *l.fit = -1;
        (void)cudaGetLastError();
        return cudaSuccess;
    }
    return cudaLaunchKernelEx(&l.cfg, kernel, (const unsigned char*)c->kimp, c->geom, ut, order, a, l.room, l.most, l.keep_scores, c->st.idx, c->st.cnt, c->st.status);
}

template <int kThreads>
cudaError_t launch_any(const tb_ctx* c, const UnitTable& ut, const StreamOrder& order, const SelectArgs& a, const StreamLaunch& l) {
    const bool max = a.reduce == TB_GROUP_MAX, wide = c->geom.dp == 32;
#define TB_STREAM(T)                                                                                                                    \
    (wide ? max ? launch<T, 32, TB_GROUP_MAX, kThreads>(c, ut, order, a, l) : launch<T, 32, TB_GROUP_SUM, kThreads>(c, ut, order, a, l) \
          : max ? launch<T, 16, TB_GROUP_MAX, kThreads>(c, ut, order, a, l) : launch<T, 16, TB_GROUP_SUM, kThreads>(c, ut, order, a, l))
    return c->geom.dtype == TB_BF16 ? TB_STREAM(__nv_bfloat16) : TB_STREAM(float);
#undef TB_STREAM
}

}  // namespace

cudaError_t launch_select_stream(const tb_ctx* c, const UnitTable& ut, const SelectArgs& a_in, cudaStream_t s, bool dry, bool* taken) {
    const Geom& gm = c->geom;
    const int n_units = ut.layer_count * ut.n_seq * gm.Hl;
    *taken = false;
    const int n_pairs = ut.layer_count * ut.n_seq;
    WaveOrder longest;
    int cand[kMaxLaunchUnits];
    const int max_cand = longest_first(ut, a_in, longest, cand);
    StreamOrder order;
    for (int i = 0; i < n_pairs; ++i) order.pair[i] = (uint16_t)(longest.pair[i] / ut.n_seq << 8 | longest.pair[i] % ut.n_seq);
    SelectArgs a = a_in;
    a.dst_is_state = 1, a.idx_dst = a.cnt_dst = nullptr, a.idx_stride = gm.idx_cap;
    StreamLaunch l = {};
    l.cfg.blockDim = dim3(512, 1, 1), l.cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
    l.cfg.attrs = attr, l.cfg.numAttrs = 1;
    // how many clusters of C blocks run at once: one block per SM, whatever its shared memory
    auto fits = [&](int C) {
        if (C == 1) return c->sm_count;
        return clusters_that_fit(C, [&] {
            attr[0].val.clusterDim.x = C;
            int n = -1;
            l.cfg.gridDim = dim3(C, 1, 1), l.cfg.dynamicSmemBytes = 100 * 1024, l.fit = &n;
            if (launch_any<512>(c, ut, order, a, l) != cudaSuccess) n = -1;
            l.fit = nullptr;
            return n;
        });
    };
    // Up to a problem per SM: blocks of 512 threads, as many per problem as run at once, each with at least 1024 rows.  us per
    // launch, bf16, 32 dimensions, a tenth selected, against the kernels before (clusters on TMA rings): 8 problems of 131072
    // candidates 25.3 / 41.2, 16 of 131072 35 / 75, 32 of 32768 20.0 / 21.5, 48 of 12000 15.7 / 24.7, 64 of 49152 42.8 / 58, 96 of
    // 32768 44 / 60, 16 of 65536 with neighbours 42 / 70.
    // More problems: one block of 256 threads each, two per SM, so that one's finish runs beside the other's stream (160 of 12000:
    // 31.6, 40.7 with 512 threads, 41.1 before; 256 of 24000 72 / 76 / 87).  Beyond two per SM the kernel that keeps four blocks
    // per SM resident has no last wave; this one wins where its own is full (512 problems, 86 %: 12000 74 / 81, 24000 137 / 156,
    // ragged 8192 to 16384 66 / 70; 8000 55 / 58 but ragged 47 / 46; 384, 65 %: 12000 68 / 65) and scoring heads one by one or two
    // problems' worth of rows per line (16 dimensions) is what the other spends its time on.  fp32 rows: 256 of 8000 53 / 62, 512
    // of 12000 137 / 153, but 160 of 12000 59 / 50 and 160 of 40000 219 / 210.
    int C = 1;
    const int sms = c->sm_count;
    int threads = n_units <= sms ? 512 : 256;
    if (n_units <= sms) {
        const int sizes[] = {16, 12, 10, 9, 8, 6, 5, 4, 3, 2, 1};
        for (int x : sizes) {
            C = x;
            if (max_cand >= 1024 * x && n_units * x <= sms && fits(x) >= n_units) break;
        }
    } else {
        const bool f32 = gm.dtype != TB_BF16, max = a.reduce == TB_GROUP_MAX, narrow = gm.dp == 16;
        const int slots = 2 * sms, full = (n_units + slots - 1) / slots * slots;
        bool take;
        if (n_units <= slots) take = !f32 || max_cand <= 10 * 1024 || (2 * n_units >= 3 * sms && max_cand <= 30 * 1024);
        else if (5 * n_units >= 4 * full) take = max_cand >= (f32 || max || narrow ? 4000 : a.radius > 0 ? 16000 : 10000);
        else take = !f32 && (max || narrow) && max_cand >= 16000;
        if (!take) return cudaSuccess;
    }
    // a replayed graph may find more than it declared
    const int spare = ut.use_dev_len && a.radius == 0 ? 2048 : 0;
    l.room = ((max_cand + spare + C - 1) / C + 127) / 128 * 128;
    // (neighbours: whole tiles of 256, as in the kernel of one block per list)
    l.most = a.radius > 0 ? std::min(C * l.room, (max_cand + 255) / 256 * 256) : C * l.room;
    auto smem = [&](bool scores) { return stream_smem(threads, C, l.room, a.radius > 0, scores); };
    // Two blocks of digits do not fit an SM: one of 512 threads, if two waves of them fill most of the chip (256 problems of 65536
    // 182 us, with neighbours 204, 230 in the kernel that parks its keys, ragged from 32768 on 144 / 187; of 50000 145 / 175).
    if (threads == 256 && smem(false) > 113 * 1024 && n_units <= 2 * sms && 4 * n_units >= 5 * sms) threads = 512;
    const int per_sm = 512 / threads;
    if ((C > 1 && l.room > kMaxShare) || smem(false) > 226 * 1024 / per_sm) return cudaSuccess;
    *taken = true;
    if (dry) return cudaSuccess;
    l.keep_scores = smem(true) <= kScoresSmem / per_sm;
    attr[0].val.clusterDim.x = C;
    l.cfg.gridDim = dim3(C, gm.Hl, n_pairs), l.cfg.blockDim = dim3(threads, 1, 1);
    l.cfg.dynamicSmemBytes = smem(l.keep_scores);
    return threads == 512 ? launch_any<512>(c, ut, order, a, l) : launch_any<256>(c, ut, order, a, l);
}

}  // namespace tb
