// Selection of small problems: scoring, exact top-B, neighbour fetching and the copy of the list for the caller, one
// block per (layer, sequence, list), one launch (paper Sec. 3.4, Sec. 4 "Token Selection Policy").
//
// A problem of a few thousand candidates is 32 KB to 1 MB of projected keys: one SM takes it in within 1 to 10 us, and
// what a launch costs beyond that is latency.  So everything stays inside one block of 512 threads; where a launch would
// leave SMs idle, up to three more blocks of a cluster stream shares of the problem into that block's shared memory:
//   stream   bf16 rows straight into tensor-core fragments (see RowStream), fp32 rows through 2-D TMA tiles of 256 rows, all
//            requested at once when they fit; the order-preserving key goes to shared memory, score sums stay in registers
//   digit    mean and deviation of all the scores place 2046 equal slices of score across mean +- 4.5 deviations (one
//            barrier), an open bin on either side; bins are monotone in the score whatever the moments say, so the
//            selection never depends on them, only how few keys share the threshold's bin does (a handful)
//   finish   histogram, threshold bin, bitmask, the bin's keys ranked pairwise (equal scores by position), neighbours
//            on the bitmask, list
// A crowded threshold bin (massive ties, a few huge outliers) goes through the key's own digits instead (11 + 11 + 10).
//
// The launch is a programmatic dependent: one block or a cluster of two or four, for which an early start finds room.
#include "tb_select.cuh"

namespace tb {

namespace {

constexpr int kHalf = 256;          // rows of a tile = threads that score it
constexpr int kBins = 2048;
constexpr int kMaxShare = 4;        // blocks that stream one problem

template <int kThreads>
struct __align__(16) SmallSmem {
    static constexpr int kWarps = kThreads / 32, kMaxCand = 32 * kThreads;   // one bitmask word per thread
    static constexpr int kMaxRank = kThreads;   // keys of the threshold bin that are ranked pairwise
    int hist[kBins];
    uint32_t mask[kMaxCand / 32], mask_out[kMaxCand / 32];
    uint2 cand[kMaxRank];           // (key, candidate) of the threshold bin
    float qs[kMaxGroup * 32];       // the list's importance queries
    uint2 frags[kQueryFrags];       // ... as tensor-core operands
    uint64_t full[kMaxCand / kHalf];
    float part[kMaxShare * kWarps][2];   // per block of the cluster and warp: sums of scores and of their squares
    int slots[kWarps];
    int bin, krem, count, n_cand;
};

__device__ __forceinline__ float key_score(uint32_t key) { return __uint_as_float(key & 0x80000000u ? key & 0x7fffffffu : ~key); }

// The bin that holds the k-th largest of the histogrammed keys: all threads get it, with k' = k - keys in higher bins
// and the bin's population.  1 <= k <= total.
template <int kThreads>
__device__ __forceinline__ void find_bin(SmallSmem<kThreads>* sm, int nbins, int k, int& bin, int& krem, int& count) {
    constexpr int kPer = kBins / kThreads, kWarps = kThreads / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int b[kPer], mine = 0;
#pragma unroll
    for (int i = 0; i < kPer; i += 4) {
        const int4 x = tid * kPer < nbins ? reinterpret_cast<const int4*>(sm->hist + tid * kPer)[i / 4] : make_int4(0, 0, 0, 0);
        b[i] = x.x, b[i + 1] = x.y, b[i + 2] = x.z, b[i + 3] = x.w;
        mine += (x.x + x.y) + (x.z + x.w);
    }
    const int incl = warp_incl_scan(mine, lane);
    if (lane == 31) sm->slots[warp] = incl;
    __syncthreads();
    int below = incl - mine, total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const int x = sm->slots[w];
        total += x;
        below += w < warp ? x : 0;
    }
    int run = total - below - mine;                    // keys in bins above this thread's
    if (run < k && k <= run + mine) {                  // exactly one thread
#pragma unroll
        for (int i = kPer - 1; i >= 0; --i) {
            if (run < k && k <= run + b[i]) sm->bin = tid * kPer + i, sm->krem = k - run, sm->count = b[i];
            run += b[i];
        }
    }
    __syncthreads();
    bin = sm->bin, krem = sm->krem, count = sm->count;
}

struct NoStream {
    __device__ __forceinline__ void start(const unsigned char*, int) {}
};

// bf16 rows: kU groups of 32 rows in flight per warp (see RowStream); fp32 rows (kU = 0): through a ring of n_stages tiles.
// kShared: a cluster of blocks per problem streams it, block r the r-th run of share_tiles tiles, with keys and sums going
// to block 0's shared memory; behind one cluster barrier block 0 finishes alone.
template <typename T, int DP, int RED, int kU, bool kShared, int kThreads>
__global__ void __launch_bounds__(kThreads, kU == 2 ? 1024 / kThreads : 1) select_small_kernel(const __grid_constant__ CUtensorMap tmap,
                                                                                 const unsigned char* __restrict__ kimp, Geom gm, UnitTable ut,
                                                                                 SelectArgs a, int n_stages, int max_tiles, int share_tiles, uint32_t wait_limit, int drop_tile,
                                                                                 int32_t* __restrict__ state_idx, int32_t* __restrict__ state_cnt,
                                                                                 int32_t* __restrict__ status) {
    constexpr int RB = DP * Elem<T>::kBytes, NCH = RB / 16;
    constexpr uint32_t kTileBytes = kHalf * RB;
    constexpr bool kDirect = kU > 0;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // swizzled boxes start on the swizzle period
    uint32_t* keys = reinterpret_cast<uint32_t*>(ring + n_stages * kTileBytes);          // max_tiles * 256
    typedef SmallSmem<kThreads> Smem;
    constexpr int kWarps = Smem::kWarps, kMaxRank = Smem::kMaxRank;
    Smem* sm = reinterpret_cast<Smem*>(keys + max_tiles * kHalf);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    uint32_t C = 1, rank = 0;
    if constexpr (kShared) {
        asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(C));
        asm volatile("mov.u32 %0, %%cluster_ctaid.x;" : "=r"(rank));
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // (waited for before the first remote store)
    }
    const int unit = blockIdx.x / C;
    // What needs nothing from the predecessor runs beside its tail.
    if (tid == 0) sm->n_cand = 0;
    if (!kDirect && warp == 0) {
        if (lane == 0) prefetch_tmap(&tmap);
        if (lane < n_stages) mbar_init(&sm->full[lane], 1), fence_mbar_init();   // (14 stages at most: 16 KB tiles)
        __syncwarp();                                  // thread 0 arms them and requests the first tiles before any block barrier
    }
    for (int i = tid; i < kBins / 4; i += kThreads) reinterpret_cast<int4*>(sm->hist)[i] = make_int4(0, 0, 0, 0);
    int ll, s, h;
    decode_unit(gm, ut, unit, ll, s, h);
    const size_t cu = list_unit(gm, ut, ll, s, h);
    const ListOut out(gm, a, cu, unit, state_idx, state_cnt);
    pdl_wait();
    pdl_launch_dependents();                           // (waits for this grid's completion before it reads a list)

    if constexpr (kShared) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");    // every block of the cluster runs
    const int L = unit_len(gm, ut, ll, s);
    const int lo = min(a.sinks, L), hi = max(lo, L - a.recent);
    const int ncand = candidates_within(hi - lo, max_tiles * kHalf, status), k = min(a.budget, ncand);
    check_candidates_projected(gm, ut, ll, s, hi, status);
    if (k <= 0 || k == ncand) {                        // nothing to rank: none, or all (neighbours add nothing then)
        if (rank == 0) out.all<kThreads>(lo, k);
        return;
    }
    const int n_tiles = (ncand + kHalf - 1) / kHalf;   // <= max_tiles
    // this block's rows: candidates slot0 .. slot0 + n_local - 1
    const int slot0 = min(ncand, (int)rank * share_tiles * kHalf), n_local = min(ncand - slot0, share_tiles * kHalf);
    const int my_tiles = (n_local + kHalf - 1) / kHalf;
    const long long row0 = (long long)key_unit(gm, ut, ll, s, h) * gm.max_seq_len + lo + slot0;
    auto request = [&](int t) {                        // tile t, into its stage
        uint64_t* bar = &sm->full[t % n_stages];
        mbar_arrive_expect_tx(bar, kTileBytes);
        // drop_tile: diagnostics only (see tb_set_wait_diagnostics): the barrier is armed and the copy left out
        if (t != drop_tile) tma_load_2d(ring + t % n_stages * kTileBytes, &tmap, 0, (int)(row0 + (long long)t * kHalf), bar);
    };
    if (!kDirect && tid == 0)
        for (int t = 0; t < min(n_stages, my_tiles); ++t) request(t);
    if (tid < gm.gl * DP) sm->qs[tid] = a.q_imp[query_row(gm, ut, ll, s, h) * DP + tid];
    typename std::conditional<kDirect, RowStream<FragScorer<DP, RED>, kDirect ? kU : 1, kWarps>, NoStream>::type rs;
    rs.start(kimp + row0 * RB, n_local);
    const bool odd_query = __syncthreads_or(kDirect && tid < gm.gl * DP && !is_finite(sm->qs[tid]));   // (its own element)

    // ---- stream ------------------------------------------------------------------------------------
    float s1 = 0.f, s2 = 0.f;
    uint32_t keys0 = smem_u32(keys + slot0), part0 = smem_u32(&sm->part[rank * kWarps + warp]);
    if constexpr (kShared) {                           // the same places in block 0
        asm volatile("mapa.shared::cluster.u32 %0, %0, 0;" : "+r"(keys0));
        asm volatile("mapa.shared::cluster.u32 %0, %0, 0;" : "+r"(part0));
    }
    auto put_key = [&](int slot, uint32_t key) {
        if constexpr (kShared) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(keys0 + slot * 4), "r"(key) : "memory");
        else keys[slot] = key;
    };
    auto keep = [&](int slot, float sc) {
        put_key(slot, order_key(sc));
        s1 += sc, s2 = fmaf(sc, sc, s2);
    };
    if constexpr (kDirect) {
        FragScorer<DP, RED> scorer;
        scorer.load_staged(sm->qs, gm.gl, sm->frags);
        rs.run(scorer, keep);
        if (odd_query || !is_finite(s1))               // infinite scores, or scores dropped beside an infinite query (see FragScorer)
            rs.own_rows([&](int slot) {
                const float sc = rescore<DP, RED>(rs.rows + (size_t)slot * RB, sm->qs, gm.gl);
                if (!is_finite(sc)) put_key(slot, order_key(sc));
            });
    } else {
        // The two halves of the block take tiles in turn; the number of stages is even when stages are used again, so that
        // a stage belongs to one half (its barrier's phases are then waited for in order).  A wait that runs out
        // (wait_limit polls; a correct run never gets there) makes its half request nothing further, score what it never
        // received as the lowest key and go on; the other half's waits are bounded the same way, so every copy in flight
        // has landed or been waited for in full before the block ends.
        GroupScorer<T, DP, RED> scorer;
        scorer.load_staged(sm->qs, gm.gl);
        const int half = tid / kHalf, r = tid % kHalf;
        bool dead = false;
        for (int t = half; t < my_tiles; t += 2) {
            const int st = t % n_stages, slot = t * kHalf + r;
            const bool ok = mbar_wait(&sm->full[st], (t / n_stages) & 1, wait_limit);
            dead |= !ok;
            const unsigned char* tile = ring + st * kTileBytes;
            if (slot < n_local && ok) {
                const uint32_t off = r * RB;
                keep(slot, scorer.score([&](int c) {
                    uint32_t o = off + c * 16;
                    o ^= ((o >> 7) & (NCH - 1)) << 4;  // TMA swizzle of 16-byte chunks (mode = row size)
                    return *reinterpret_cast<const uint4*>(tile + o);
                }));
            } else if (slot < n_local) {
                put_key(slot, 0u);
            }
            if (t + n_stages < my_tiles) {             // uniform per half
                if (half == 0) asm volatile("bar.sync 1, %0;" ::"n"(kHalf) : "memory");   // the half has read the stage
                else asm volatile("bar.sync 2, %0;" ::"n"(kHalf) : "memory");
                if (r == 0 && !dead) {
                    fence_proxy_async();
                    request(t + n_stages);
                }
            }
        }
        if (dead && lane == 0) atomicExch(status, kStatusTimeout);
    }
    s1 = warp_sum(s1), s2 = warp_sum(s2);
    if constexpr (kShared) {
        if (lane == 0) {
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(part0), "f"(s1) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(part0 + 4), "f"(s2) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank != 0) return;                         // nothing reads this block's shared memory
    } else {
        if (lane == 0) sm->part[warp][0] = s1, sm->part[warp][1] = s2;
        __syncthreads();
    }

    // ---- digit and histogram --------------------------------------------------------------------------
    float m1 = 0.f, m2 = 0.f;
    for (int r = 0; r < (int)C; ++r)
#pragma unroll
        for (int w = 0; w < kWarps; ++w) m1 += sm->part[r * kWarps + w][0], m2 += sm->part[r * kWarps + w][1];
    m1 /= (float)ncand, m2 = m2 / (float)ncand - m1 * m1;
    const float dev = sqrtf(fmaxf(m2, 0.f));
    const float base = m1 - 4.5f * dev, scale = dev > 0.f ? (float)(kBins - 2) / (9.f * dev) : 0.f;
    auto bin_of = [&](uint32_t key) { return (int)fminf(fmaxf((key_score(key) - base) * scale + 1.f, 0.f), (float)(kBins - 1)); };
    for (int i = tid; i < ncand; i += kThreads) atomicAdd(&sm->hist[bin_of(keys[i])], 1);
    __syncthreads();
    int bin, kr, bc;
    find_bin(sm, kBins, k, bin, kr, bc);

    const uint4* keys4 = reinterpret_cast<const uint4*>(keys);
    // verdict(key): 2 = selected, 1 = to be ranked among its equals-so-far, 0 = not.  Lane l of a warp holds slots
    // 4 l .. 4 l + 3 of a group: its verdicts are a nibble of the bitmask, eight lanes make a word.
    auto classify = [&](auto verdict, bool whole) {
        for (int v = tid; v < n_tiles * (kHalf / 4); v += kThreads) {
            const uint4 x = keys4[v];
            const uint32_t kk[4] = {x.x, x.y, x.z, x.w};
            uint32_t word = 0u, rank = 0u;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int w = v * 4 + e < ncand ? verdict(kk[e]) : 0;
                word |= (uint32_t)(w == 2 || (whole && w == 1)) << e;
                rank |= (uint32_t)(w == 1 && !whole) << e;
            }
            word <<= 4 * (lane & 7);
            word |= __shfl_xor_sync(0xffffffffu, word, 1);
            word |= __shfl_xor_sync(0xffffffffu, word, 2);
            word |= __shfl_xor_sync(0xffffffffu, word, 4);
            if ((lane & 7) == 0) sm->mask[v >> 3] = word;
            while (rank) {
                const int e = __ffs(rank) - 1;
                rank &= rank - 1;
                sm->cand[atomicAdd(&sm->n_cand, 1)] = make_uint2(keys[v * 4 + e], (uint32_t)(v * 4 + e));
            }
        }
        __syncthreads();
    };
    if (bc == kr || bc <= kMaxRank) {
        classify([&](uint32_t key) { const int b = bin_of(key); return b > bin ? 2 : b == bin ? 1 : 0; }, bc == kr);
        if (bc != kr) {
            if (tid < bc) {                            // rank: larger key first, equal keys by position
                const uint2 it = sm->cand[tid];
                int before = 0;
#pragma unroll 4
                for (int j = 0; j < bc; ++j) {
                    const uint2 o = sm->cand[j];
                    before += (o.x > it.x) | ((o.x == it.x) & (o.y < it.y));
                }
                if (before < kr) atomicOr(&sm->mask[it.y >> 5], 1u << (it.y & 31));
            }
            __syncthreads();
        }
    } else {
        // The key's own digits.  What is left at the end are equal keys: the first ones in position order are taken.
        uint32_t prefix = 0;
        int low_bits = 32;
        kr = k;
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            const int bits = pass == 2 ? 10 : 11, shift = low_bits - bits;
            for (int i = tid; i < kBins / 4; i += kThreads) reinterpret_cast<int4*>(sm->hist)[i] = make_int4(0, 0, 0, 0);
            __syncthreads();
            for (int i = tid; i < ncand; i += kThreads) {
                const uint32_t key = keys[i];
                if (pass == 0 || (key >> low_bits) == prefix) atomicAdd(&sm->hist[(key >> shift) & ((1 << bits) - 1)], 1);
            }
            __syncthreads();
            find_bin(sm, 1 << bits, kr, bin, kr, bc);
            prefix = (prefix << bits) | (uint32_t)bin, low_bits = shift;
        }
        classify([&](uint32_t key) { return key > prefix ? 2 : 0; }, false);
        // the equal keys' bits, then as many of them as are wanted, lowest positions first
        const int n_words = n_tiles * (kHalf / 32);    // <= kThreads
        uint32_t eq = 0u;
        if (tid < n_words)
            for (int e = 0; e < 32; ++e) eq |= (uint32_t)(tid * 32 + e < ncand && keys[tid * 32 + e] == prefix) << e;
        const int n_eq = __popc(eq), incl = warp_incl_scan(n_eq, lane);
        if (lane == 31) sm->slots[warp] = incl;
        __syncthreads();
        int before = incl - n_eq;
        for (int w = 0; w < warp; ++w) before += sm->slots[w];
        uint32_t take = 0u;
        while (eq && before < kr) take |= eq & (0u - eq), eq &= eq - 1, ++before;
        if (take) sm->mask[tid] |= take;
        __syncthreads();
    }

    // ---- neighbours and list -----------------------------------------------------------------------------
    finish_mask_list<kThreads>(sm->mask, sm->mask_out, ncand, lo, out, sm->slots);
}

size_t small_smem(int n_stages, int n_tiles, int tile_bytes, int threads = 512) {
    return 1024 + (size_t)n_stages * tile_bytes + (size_t)n_tiles * kHalf * 4 + (threads == 512 ? sizeof(SmallSmem<512>) : sizeof(SmallSmem<256>));
}

}  // namespace

// As long as one block's finish is cheaper than a cluster's.  Against the streaming kernel,
// us per launch, bf16, 32 dimensions unless said (this / the other): 8 problems of 4000 candidates 7.6 / 9.8, 10000 11.1 / 11.1, 32
// of 8000 11.1 / 12.1, with neighbours 14.3 / 15.3 and 16000 20.9 / 18.5; more problems than half of the SMs leave the other
// one block each too: 96 of 8000 15.8 / 16.8, 16000 26.6 / 26.8, fp32 42.1 / 44.1; two per SM: 192 of 6000 20.6 / 21.7, 8000
// 25.4 / 26.3, with neighbours 160 of 12000 51 / 40; fp32, whose rows do not go straight into registers here, 160 of 4000 32 /
// 25, 2000 20 / 15.6.  More than two problems per SM: against the kernel of one 256-thread block each that parks its keys in memory,
// 512 of 300 8.2 / 11.6, 1000 11.6 / 15.5, 4900 36.7 / 38.8, ragged to 4900 30.7 / 32.3, 6000 42.6 / 44.1, 8000 61 / 58; 2048 of 1000 36
// / 46; lists that share a key stream, whose rows are L2 hits for all but one, 512 of 8000 41 / 47.
// Under device lengths the streaming kernel takes neither more lists than SMs nor lists that share a key stream; with neighbours,
// against the kernels that do: 160 of 9000 32 / 38, 16000 50 / 55, 296 of 16000 65 / 72, at 16 dimensions 45 / 50; one list per query
// head, four per stream, 32 of 11000 14.9 / 22.3, 16000 17.1 / 26, 160 of 9000 26.0 / 28.3, 12000 30.5 / 30.7, 16000 37 / 34.
// Whether the caller wants copies does not matter: the scores are summed in another order here, and an output that the caller
// may leave out must not decide which of two tokens within fp32 rounding of one another is stored.
bool select_small_takes(const tb_ctx* c, const UnitTable& ut, int max_cand, bool neighbours) {
    const int n_units = ut.layer_count * ut.n_seq * c->geom.Hl;
    const bool many = n_units > c->sm_count, per_head = c->geom.Hl > c->geom.Hi;
    // wait diagnostics: launches of one block that wait for copies (the others: see launch_select)
    if (c->drop_tile >= 0 && (c->geom.dtype == TB_BF16 || n_units > 1 || max_cand > 1023)) return false;
    // (Replayed graphs in which this many sequences grow: the kernel whose room is the workspace's.)
    if (n_units > 2 * c->sm_count && ut.use_dev_len) return false;
    if (many && c->geom.dtype != TB_BF16) return max_cand <= 1500;
    if (n_units > 2 * c->sm_count) return max_cand <= (per_head ? SmallSmem<256>::kMaxCand : 5000);
    if (ut.use_dev_len && neighbours && c->geom.dtype == TB_BF16 && (many || per_head))
        return max_cand <= (many && per_head ? 12 * 1024 : SmallSmem<512>::kMaxCand);
    const int most = !many ? (2 * n_units > c->sm_count ? SmallSmem<512>::kMaxCand : 10 * 1024) : 8 * 1024;
    return max_cand <= most;
}

cudaError_t launch_select_small(const tb_ctx* c, const UnitTable& ut, const SelectArgs& a, int max_cand, cudaStream_t s, bool dry) {
    if (dry) return cudaSuccess;
    const Geom& gm = c->geom;
    const int n_units = ut.layer_count * ut.n_seq * gm.Hl;
    const int tile_bytes = kHalf * gm.dp * (gm.dtype == TB_BF16 ? 2 : 4);
    const int n_tiles = max_cand > kHalf ? (max_cand + kHalf - 1) / kHalf : 1;
    const uint32_t wait_limit = c->wait_poll_limit > 0 ? (uint32_t)c->wait_poll_limit : kWaitPollLimit;
    const int drop_tile = c->drop_tile;                // one-shot
    const_cast<tb_ctx*>(c)->drop_tile = -1;

    // fp32: all tiles in flight at once if an SM's share of shared memory holds them, all of it when every block has an SM
    // to itself, half otherwise.
    const bool direct = gm.dtype == TB_BF16, alone = n_units <= c->sm_count;
    const size_t room = (alone ? 226 : 112) * 1024;
    // Blocks per problem: as many as leave each at least 1024 rows and fit the SMs (a block takes in 45 to 55 bytes per clock).
    int C = 1;
    while (2 * C <= kMaxShare && 2 * C * n_units <= c->sm_count && n_tiles >= 2 * C * 4) C *= 2;
    const int share_tiles = (n_tiles + C - 1) / C;
    // Short lists, or more than fit the chip with 512 threads each: blocks of 256, four per SM (160 problems of 1000 candidates
    // 7.6 us, 8.6 with 512 threads, 2000 level, 4000 15.6 / 14.7; 512 of 1000 11.5 / 17.1).
    const int threads = direct && (n_units > 2 * c->sm_count || (!alone && max_cand <= 2048)) ? 256 : 512;
    int n_stages = direct ? 0 : share_tiles;
    if (small_smem(n_stages, n_tiles, tile_bytes) > room) {
        n_stages &= ~1;                                // even: see the stream loop
        while (n_stages > 2 && small_smem(n_stages, n_tiles, tile_bytes) > room) n_stages -= 2;
    }

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_units * C, 1, 1), cfg.blockDim = dim3(threads, 1, 1), cfg.stream = s;
    cfg.dynamicSmemBytes = small_smem(n_stages, n_tiles, tile_bytes, threads);
    cudaLaunchAttribute attr[2];
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = C, attr[1].val.clusterDim.y = 1, attr[1].val.clusterDim.z = 1;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see pdl_wait()
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr, cfg.numAttrs = C > 1 ? 2 : 1;
    auto launch = [&](auto kernel, DeviceFlags& done) {
        const cudaError_t e = allow_shared_memory(done, kernel, 227 * 1024);
        if (e != cudaSuccess) return e;
        return cudaLaunchKernelEx(&cfg, kernel, c->kimp_map, (const unsigned char*)c->kimp, gm, ut, a, n_stages, n_tiles, share_tiles, wait_limit, drop_tile,
                                  c->st.idx, c->st.cnt, c->st.status);
    };
    // a block alone on its SM keeps four groups of rows in flight per warp, two blocks two each (their registers)
#define TB_SMALL(T, DP, RED, U, SH, NT)                                    \
    do {                                                                   \
        static DeviceFlags done;                                           \
        return launch(select_small_kernel<T, DP, RED, U, SH, NT>, done);   \
    } while (0)
#define TB_SMALL_U(DP, RED)                                                      \
    do {                                                                         \
        if (direct && C > 1) TB_SMALL(__nv_bfloat16, DP, RED, 4, true, 512);     \
        if (direct && alone) TB_SMALL(__nv_bfloat16, DP, RED, 4, false, 512);    \
        if (direct && threads == 256) TB_SMALL(__nv_bfloat16, DP, RED, 2, false, 256); \
        if (direct) TB_SMALL(__nv_bfloat16, DP, RED, 2, false, 512);             \
        if (C > 1) TB_SMALL(float, DP, RED, 0, true, 512);                       \
        TB_SMALL(float, DP, RED, 0, false, 512);                                 \
    } while (0)
    const bool max = a.reduce == TB_GROUP_MAX;
    if (gm.dp == 32) {
        if (max) TB_SMALL_U(32, TB_GROUP_MAX);
        TB_SMALL_U(32, TB_GROUP_SUM);
    }
    if (max) TB_SMALL_U(16, TB_GROUP_MAX);
    TB_SMALL_U(16, TB_GROUP_SUM);
#undef TB_SMALL_U
#undef TB_SMALL
}

}  // namespace tb
