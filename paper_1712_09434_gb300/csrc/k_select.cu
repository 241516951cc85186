// S6 track selection: the exact result of the sequential greedy rule, computed in parallel rounds.
//
// Sequential rule: candidates in priority order (more hits first, then earlier seed) keep the hits
// that no already-accepted candidate owns and are accepted with at least N_MIN kept hits.  Hits
// belong to one sector, so an (event, sector) is one item.  Priority key (unique, smaller =
// earlier): ((n_rows - n_hits) << 23) | (candidate index in the sector).
//
// Every cluster has one 64-bit word: 0, (round << 32 | ~key) of the latest round's smallest key
// that claims it, or (~0 << 32 | ~key) once the accepted candidate `key` owns it.  Round: every
// undecided candidate claims its hits (atomicMax); an undecided candidate whose hits are all
// resolved (owned = lost, or claimed by itself = kept) decides, and if accepted takes ownership of
// its kept hits at once; one that cannot reach N_MIN even with its unresolved hits is rejected.
// The highest-priority undecided candidate always decides, so the rounds end, and every decision
// equals the sequential one (a candidate decides only when no higher-priority undecided candidate
// shares a hit with it).  The kept hits of an accepted candidate are written as a bit per row of
// its row range, which is all that the merge and the track output read afterwards.
//
// What bounds it: the dependent loads of a candidate (its list entry, its row slots, their words)
// and the barriers of a round.  A round only touches the undecided candidates: they are kept as a
// compact list (candidate, key, rows) per block, read ahead of its use with the candidate's row
// slots, and from the second round on a candidate that has lost its hits is dropped before it
// claims any.
#include "tpc_common.cuh"

namespace tpc {

namespace {

constexpr int SEL_ILP = 5;   // row slots per lane loaded before their dependent loads (5 x 32 >= 159)
constexpr uint32_t SEL_OWNED = 0xffffffffu;   // round tag of an owned hit (rounds stay below 2^14)

__device__ __forceinline__ uint32_t key_of(int n_rows, int n_hits, int local) {
    return ((uint32_t)(n_rows - n_hits) << 23) | (uint32_t)local;
}

// Barrier of the blocks that share an item: release / acquire at the scope of the group.  Every thread
// arrives on its own (no .aligned): the loops before it end at different times for the lanes of a
// warp, and nothing but the compiler would bring them together again.
template <int CS>
__device__ __forceinline__ void group_sync() {
    if constexpr (CS == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
    }
}

template <int CS>
__device__ __forceinline__ int group_rank() {
    if constexpr (CS == 1) return 0;
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}

// value of the shared word `p` of block `rank` of the group
template <int CS>
__device__ __forceinline__ int group_read(const int *p, int rank) {
    if constexpr (CS == 1) return *p;
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return (int)v;
}

// A warp's walk over its entries of the candidate list, one candidate ahead: c and h are the current
// entry and this lane's row slots of it (rows row0 + lane + 32 j; -1 where there is none).
struct Ahead {
    const Work &W;
    const int4 *list;
    int n, i, step, lane, nr;
    int4 c, c1, c2;
    int h[SEL_ILP], h1[SEL_ILP];
    __device__ __forceinline__ Ahead(const Work &w, const int4 *l, int n_, int i0, int st, int ln, int r)
        : W(w), list(l), n(n_), i(i0), step(st), lane(ln), nr(r) {
        c1 = i < n ? list[i] : make_int4(-1, 0, 0, 0);
        c2 = i + step < n ? list[i + step] : make_int4(-1, 0, 0, 0);
        slots(c1, h1);
    }
    __device__ __forceinline__ void slots(const int4 &e, int *x) const {
        const int32_t *sl = W.cand_slots + (size_t)e.x * nr;
        const int rb = e.z >> 16;
#pragma unroll
        for (int j = 0; j < SEL_ILP; j++) {
            const int r = (e.z & 0xffff) + lane + 32 * j;
            x[j] = e.x >= 0 && r <= rb ? sl[r] : -1;
        }
    }
    __device__ __forceinline__ void next() {
        c = c1;
#pragma unroll
        for (int j = 0; j < SEL_ILP; j++) h[j] = h1[j];
        c1 = c2;
        i += step;
        c2 = i + step < n ? list[i + step] : make_int4(-1, 0, 0, 0);
        slots(c1, h1);
    }
};

// CS blocks (a thread-block cluster) take one item together, each with its own share of the
// candidates; inside a block a warp takes one candidate at a time, its lanes the row slots.
template <int CS>
__global__ void __launch_bounds__(1024) k_select(Work W) {
    __shared__ int s_item, s_cnt[3];
    const DevGeom &g = *W.geom;
    const int nr = g.n_rows, ns = g.n_sectors;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int rank = group_rank<CS>();
    int n_chains = W.counters[CNT_NCHAINS];
    if (n_chains > W.cap_chains) n_chains = W.cap_chains;
    const int n_items = W.n_events * ns;
    int32_t *q = W.counters + CNT_Q0 + 4;
    unsigned long long *claim = reinterpret_cast<unsigned long long *>(W.claim);
    const int kw = kept_words(nr);
    // one block an item: from the queue; a cluster an item: in turn (every cluster has about one)
    int it = CS == 1 ? queue_next(q, 1, &s_item) : (int)(blockIdx.x / CS);
    for (; it < n_items; it = CS == 1 ? queue_next(q, 1, &s_item) : it + (int)(gridDim.x / CS)) {
        const int b0 = it * nr;   // (event*ns + sector)*nr
        const int t0 = min(W.chain_off[b0], n_chains), t1 = min(W.chain_off[b0 + nr], n_chains);
        const int cl0 = W.bin_off[b0], cl1 = W.bin_off[b0 + nr];
        for (int c = cl0 + rank * (int)blockDim.x + (int)threadIdx.x; c < cl1; c += CS * blockDim.x) claim[c] = 0ull;
        if (threadIdx.x < 3) s_cnt[threadIdx.x] = 0;
        __syncthreads();
        // this block's candidates (every CS-th of the item) that can be accepted at all, as a list; a
        // candidate with fewer than N_MIN hits never claims (the sequential rule gives it nothing
        // either).  The lists live in the merge's segment ends, which are written after this kernel.
        const int per = (t1 - t0) / CS, rest = (t1 - t0) % CS;
        const int share = per + (rank < rest ? 1 : 0);
        int4 *cur = W.outend + t0 + rank * per + min(rank, rest), *nxt = cur + (W.cap_chains + 1);
        for (int i = (int)threadIdx.x; i < share; i += blockDim.x) {
            const int t = t0 + i * CS + rank;
            const int n = W.cand_n[t];
            W.seg_n[t] = 0;
            if (n < N_MIN) continue;
            cur[atomicAdd(&s_cnt[0], 1)] = make_int4(t, (int)key_of(nr, n, t - t0), W.cand_rows[t], 0);
        }
        group_sync<CS>();
        int n_cur = s_cnt[0];
        int round = 1;
        bool more = true;
        for (; more && round <= SELECT_MAX_ROUNDS; round++) {
            // counters in turn: this round's, and the next one's, whose last readers are two rounds back
            int *cnt = &s_cnt[round % 3];
            if (threadIdx.x == 0) s_cnt[(round + 1) % 3] = 0;
            // Claims.  From the second round on a candidate first looks at its hits: with fewer than
            // N_MIN of them unowned it is rejected here, and it claims only the unowned ones.  The row
            // slots of the next candidate are loaded while this one's words are on their way.
            Ahead A(W, cur, n_cur, warp, nwarps, lane, nr);
            for (int i = warp; i < n_cur; i += nwarps) {
                A.next();
                const int4 c = A.c;
                const unsigned long long v = ((unsigned long long)round << 32) | (uint32_t)~(uint32_t)c.y;
                const int ra = c.z & 0xffff, rb = c.z >> 16;
                if (round == 1) {
#pragma unroll
                    for (int j = 0; j < SEL_ILP; j++)
                        if (A.h[j] >= 0) atomicMax(claim + A.h[j], v);
                    for (int r = ra + 32 * SEL_ILP + lane; r <= rb; r += 32) {     // more than 160 rows
                        const int h = W.cand_slots[(size_t)c.x * nr + r];
                        if (h >= 0) atomicMax(claim + h, v);
                    }
                    continue;
                }
                unsigned long long cv[SEL_ILP];
                int open = 0;
#pragma unroll
                for (int j = 0; j < SEL_ILP; j++) cv[j] = A.h[j] >= 0 ? __ldcg(claim + A.h[j]) : ~0ull;
#pragma unroll
                for (int j = 0; j < SEL_ILP; j++)
                    open += __popc(__ballot_sync(0xffffffffu, (uint32_t)(cv[j] >> 32) != SEL_OWNED));
                for (int r0 = ra + 32 * SEL_ILP; r0 <= rb; r0 += 32) {
                    const int r = r0 + lane;
                    const int h = r <= rb ? W.cand_slots[(size_t)c.x * nr + r] : -1;
                    const bool o = h >= 0 && (uint32_t)(__ldcg(claim + h) >> 32) != SEL_OWNED;
                    open += __popc(__ballot_sync(0xffffffffu, o));
                    if (o) atomicMax(claim + h, v);
                }
                if (open < N_MIN) {
                    if (lane == 0) cur[i].x = -1;
                    continue;
                }
#pragma unroll
                for (int j = 0; j < SEL_ILP; j++)
                    if ((uint32_t)(cv[j] >> 32) != SEL_OWNED) atomicMax(claim + A.h[j], v);
            }
            group_sync<CS>();
            // Decisions.  A candidate accepted in this round takes ownership of its kept hits at once:
            // only the claimant of a hit can own it, and a later reader that already sees the owner
            // counts the hit as lost, which is the sequential answer for it (its owner is accepted).
            Ahead B(W, cur, n_cur, warp, nwarps, lane, nr);
            for (int i = warp; i < n_cur; i += nwarps) {
                B.next();
                const int4 c = B.c;
                if (c.x < 0) continue;                       // rejected above
                const unsigned long long v = ((unsigned long long)round << 32) | (uint32_t)~(uint32_t)c.y;
                const int ra = c.z & 0xffff, rb = c.z >> 16;
                const int32_t *sl = W.cand_slots + (size_t)c.x * nr;
                int sure = 0, unk = 0;
                unsigned mine = 0;                           // bit j: this lane's slot j is kept
                unsigned long long cv[SEL_ILP];
#pragma unroll
                for (int j = 0; j < SEL_ILP; j++) cv[j] = B.h[j] >= 0 ? __ldcg(claim + B.h[j]) : ~0ull;
#pragma unroll
                for (int j = 0; j < SEL_ILP; j++) {
                    const bool m = cv[j] == v;
                    if (m) mine |= 1u << j;
                    sure += __popc(__ballot_sync(0xffffffffu, m));
                    unk += __popc(__ballot_sync(0xffffffffu, !m && (uint32_t)(cv[j] >> 32) != SEL_OWNED));
                }
                for (int r0 = ra + 32 * SEL_ILP; r0 <= rb; r0 += 32) {
                    const int r = r0 + lane;
                    const int h = r <= rb ? sl[r] : -1;
                    const unsigned long long x = h >= 0 ? __ldcg(claim + h) : ~0ull;
                    sure += __popc(__ballot_sync(0xffffffffu, x == v));
                    unk += __popc(__ballot_sync(0xffffffffu, x != v && (uint32_t)(x >> 32) != SEL_OWNED));
                }
                if (unk == 0) {
                    if (sure >= N_MIN) {
                        const unsigned long long own = ((unsigned long long)SEL_OWNED << 32) | (uint32_t)~(uint32_t)c.y;
                        uint32_t *km = W.kept + (size_t)c.x * kw;
#pragma unroll
                        for (int j = 0; j < SEL_ILP; j++) {
                            const bool k = (mine >> j) & 1u;
                            const unsigned m = __ballot_sync(0xffffffffu, k);
                            if (k) claim[B.h[j]] = own;
                            if (lane == j && j < kw) km[j] = m;
                        }
                        for (int r0 = ra + 32 * SEL_ILP; r0 <= rb; r0 += 32) {
                            const int r = r0 + lane;
                            const int h = r <= rb ? sl[r] : -1;
                            const bool k = h >= 0 && __ldcg(claim + h) == v;
                            const unsigned m = __ballot_sync(0xffffffffu, k);
                            if (k) claim[h] = own;
                            if (lane == 0) km[(r0 - ra) >> 5] = m;
                        }
                        if (lane == 0) W.seg_n[c.x] = sure;
                    }
                } else if (sure + unk >= N_MIN && lane == 0) {
                    nxt[atomicAdd(cnt, 1)] = c;            // undecided: next round
                }
            }
            group_sync<CS>();
            n_cur = *cnt;
            int all = n_cur;
            if constexpr (CS > 1) {
                all = 0;
#pragma unroll
                for (int k = 0; k < CS; k++) all += group_read<CS>(cnt, k);
            }
            more = all != 0;
            int4 *x = cur;
            cur = nxt;
            nxt = x;
        }
        round -= 1;
        if (threadIdx.x == 0) {
            if (more) set_status(W, ST_TIMEOUT);      // left undecided: no kept hits
            atomicMax(W.counters + CNT_ROUNDS, round);
        }
        group_sync<CS>();      // the counters are reused, and another block may still read them
    }
}

template <int CS>
void launch_cluster(const Work &W, int items, int block, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(items * CS);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_select<CS>, W);
}

}  // namespace

// Blocks that share an item.  A group of 2 or 4 spreads a sector over more multiprocessors (one
// block of 1024 threads each) and is taken where it clearly shortens the waves of blocks over them:
// one event (36 items) 4 blocks each, the five dense slices of a time frame (180 items) 4, batches
// of many events 1.  Measured, one / two / four blocks an item: central event 885 / 507 / 320 us (a
// single block that scans all candidate states every round 1285 us), 5,000-track event 110 / 88 /
// 74, 5 slices 1005 / 682 / 646 (1460), 12 events 115 / 167 / 229, 64 events 2.14 / 2.52 / 3.39 ms
// (2.65); groups of 8 were behind 4 everywhere.  A launch shape with a grid of its own (ctas_per_sm)
// takes one block an item.
int group_size(int items, int block, int sm_count) {
    const int slots = sm_count * (1024 / block);
    int cs = 1;
    float best = 0.f;
    for (int k = 1; k <= 4; k *= 2) {
        const float waves = (float)((items * k + slots - 1) / slots) / k;
        if (k == 1 || waves < 0.85f * best) { best = waves; cs = k; }
    }
    return cs;
}

void launch_select(const Work &W, cudaStream_t s) {
    const int block = W.tune.block[4] > 0 ? W.tune.block[4] : 1024;
    const int items = W.n_events * W.ns;
    const int cs = W.tune.grid[4] > 0 ? 1 : group_size(items, block, W.sm_count);
    if (cs == 4) {
        launch_cluster<4>(W, items, block, s);
    } else if (cs == 2) {
        launch_cluster<2>(W, items, block, s);
    } else {
        int grid = W.tune.grid[4] > 0 ? W.tune.grid[4] : W.sm_count * 2;
        if (grid > items) grid = items > 0 ? items : 1;
        k_select<1><<<grid, block, 0, s>>>(W);
    }
}

}  // namespace tpc
