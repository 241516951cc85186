// S5 track following: Kalman-filter following of each seed across the pad rows (arxiv 1712.09434
// section 3).  Every accept/reject decision is taken by an integer steady-state Kalman filter (abg.cuh:
// alpha-beta-gamma = 1/2, 1/8, 1/32 on a Q16 state, floor shifts) so that the hit lists are
// bit-identical to an independent FP64 implementation; the floating-point Kalman filter is used for
// the parameters only (S8).
//
// A chain is followed by two threads at once: one filters along it in ascending rows and extends it
// row by row outwards, the other filters in descending rows and extends it inwards.  A step: predict,
// look up the nearest cluster (minimum (d^2, index)) within a radius that grows with consecutive
// misses in the row's Z-slab grid, update.  A candidate is stored as one cluster per row (-1 for a
// miss) between its first and last row.  The chains are taken in an order that groups chains of equal
// length and nearby start rows in a warp (below).
//
// What bounds it: the dependent loads of one thread's steps (link, coordinates; slab offsets, search)
// and the instructions of a divergent search, over the threads in flight.  Two threads a chain halve
// the serial length, the filter runs in 32-bit words where the geometry allows it, which also leaves
// registers for ten blocks of 128 threads a multiprocessor, and the row offset and the found
// cluster's index are off the step's critical path.  Measured (one thread a chain with a 64-bit
// filter -> this): 64 events of 1.14 M chains 4.15 -> 3.02 ms, a central event 861 -> 643 us, a
// 5,000-track event 446 -> 360 us, one sector of 138 chains 350 -> 190 us; with the 64-bit filter
// 3.79 ms, 746, 331 and 213 us.  Reading a slab four entries at a time instead of by binary search
// was slower where rows are dense (4.0 ms, 802 us).
#include "abg.cuh"
#include "tpc_common.cuh"

namespace tpc {

namespace {

__device__ __forceinline__ int slab_of(int z) { int s = z >> ZB_SHIFT; return s < NZB - 1 ? s : NZB - 1; }

// Nearest cluster of a row (its grid entries yz, indices loc, slab offsets zo) to (py, pz) with
// d^2 <= w^2 (w < 512): its position in the row's grid, or -1; its packed (Y, Z) goes to *yz_out
// (the cluster arrays need not be read again).  Of equal distances the smallest index counts.
__device__ __forceinline__ int nearest(const int32_t *yz, const uint16_t *loc, const uint16_t *zo, int py, int pz,
                                       int w, int32_t *yz_out) {
    const int zl = slab_of(max(pz - w, 0)), zh = slab_of(pz + w);
    const int w2 = w * w;
    int bd = w2 + 1, bi = -1;
    int32_t bv = 0;
    for (int s = zl; s <= zh; s++) {
        int a = __ldg(zo + s), e = __ldg(zo + s + 1);
        const int hi = e;
        while (a < e) {
            const int mid = (a + e) >> 1;
            if (grid_y(__ldg(yz + mid)) < py - w) a = mid + 1; else e = mid;
        }
        for (int i = a; i < hi; i++) {
            const int32_t v = __ldg(yz + i);
            const int dy = grid_y(v) - py;
            if (dy > w) break;
            const int dz = grid_z(v) - pz;
            if (abs(dz) > w) continue;
            const int d2 = dy * dy + dz * dz;
            if (d2 < bd || (d2 == bd && d2 <= w2 && __ldg(loc + i) < __ldg(loc + bi))) { bd = d2; bi = i; bv = v; }
        }
    }
    *yz_out = bv;
    return bi;
}

// Extend from the filter state (already at row `row_last`) in direction dir; writes slots.
// Returns the number of clusters found and the row of the last one in *row_end.  The next row's
// cluster offset is loaded during a row, and a found cluster's index is stored during the next one.
template <class T>
__device__ __forceinline__ int extend(const Work &W, const DevGeom &g, Abg<T> &fy, Abg<T> &fz, int rowbase_bin,
                                      int row_last, int dir, int nr, int32_t *slots, int *row_end) {
    int n = 0, misses = 0;
    *row_end = row_last;
    int row = row_last + dir;
    int c_next = 0, pend = -1, pend_row = -1;      // a found cluster not stored yet
    if (row >= 0 && row < nr) c_next = __ldg(W.bin_off + rowbase_bin + row);
    while (row >= 0 && row < nr) {
        const int c0 = c_next;
        abg_predict(fy);
        abg_predict(fz);
        const int py = q16_round(fy.p), pz = q16_round(fz.p) + Abg<T>::ZB;
        if (abs(py) > g.ymax[row] || pz < 0 || pz > g.zmax || fy.v > (T)V_MAX * 65536 || fy.v < -(T)V_MAX * 65536) break;
        const int w = W_F0 + W_F1 * misses;
        const int bin = rowbase_bin + row;
        if (row + dir >= 0) c_next = __ldg(W.bin_off + bin + dir);
        const int ps = pstart_of(c0, bin);
        int32_t v;
        const int i = nearest(W.gyz + ps, W.gloc + ps, W.zoff + (size_t)bin * ZOFF_STRIDE, py, pz, w, &v);
        if (pend_row >= 0) slots[pend_row] = pend;
        if (i >= 0) {
            pend = c0 + (int)__ldg(W.gloc + ps + i);
            pend_row = row;
            abg_update(fy, grid_y(v));
            abg_update(fz, grid_z(v) - Abg<T>::ZB);
            *row_end = row;
            n++;
            misses = 0;
        } else {
            pend_row = -1;
            slots[row] = -1;
            if (++misses >= M_MISS) break;
        }
        row += dir;
    }
    if (pend_row >= 0) slots[pend_row] = pend;
    return n;
}

// Order in which the following takes the chains: per (event, sector), by groups of 16 start rows
// and inside a group by decreasing chain length (lengths of 127 and more together), so that the
// lanes of a warp filter chains of about the same length from about the same row and leave the
// chain at about the same time.  One block per (event, sector): a counting sort in shared memory.
// The candidates are still written at the chains' own indices, so the order changes no result.
constexpr int FO_ROWS = 16, FO_LEN = 128, FO_KEYS = (MAX_ROWS / FO_ROWS) * FO_LEN;
__global__ void __launch_bounds__(256) k_follow_order(Work W, int32_t *perm) {
    __shared__ int s_cnt[FO_KEYS];
    const int nr = W.geom->n_rows, ns = W.geom->n_sectors;
    int n_chains = W.counters[CNT_NCHAINS];
    if (n_chains > W.cap_chains) n_chains = W.cap_chains;
    const int nkeys = ((nr + FO_ROWS - 1) / FO_ROWS) * FO_LEN;
    for (int it = blockIdx.x; it < W.n_events * ns; it += gridDim.x) {
        const int b0 = it * nr;
        const int t0 = min(W.chain_off[b0], n_chains), t1 = min(W.chain_off[b0 + nr], n_chains);
        if (t1 <= t0) continue;      // the same for the whole block
        for (int k = threadIdx.x; k < nkeys; k += blockDim.x) s_cnt[k] = 0;
        __syncthreads();
        for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
            const int key = ((W.chain_bin[t] - b0) / FO_ROWS) * FO_LEN + (FO_LEN - 1 - min(W.chain_len[t], FO_LEN - 1));
            atomicAdd(&s_cnt[key], 1);
        }
        __syncthreads();
        if (threadIdx.x < 32) {      // exclusive scan of the counts by one warp, in key order
            int run = t0;
            for (int k0 = 0; k0 < nkeys; k0 += 32) {
                const int k = k0 + threadIdx.x;
                const int v = k < nkeys ? s_cnt[k] : 0;
                int x = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (threadIdx.x >= o) x += y;
                }
                if (k < nkeys) s_cnt[k] = run + x - v;
                run += __shfl_sync(0xffffffffu, x, 31);
            }
        }
        __syncthreads();
        for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
            const int key = ((W.chain_bin[t] - b0) / FO_ROWS) * FO_LEN + (FO_LEN - 1 - min(W.chain_len[t], FO_LEN - 1));
            perm[atomicAdd(&s_cnt[key], 1)] = t;
        }
        __syncthreads();
    }
}

// One step of the filter along the chain: `k` hits seen so far, the new one (y, z) `d` rows on.
template <class T>
struct ChainFilter {
    Abg<T> fy, fz;
    int m0y, m0z, k = 0;
    __device__ __forceinline__ void hit(int y, int z0, int d) {
        const int z = z0 - Abg<T>::ZB;
        if (k == 0) {
            m0y = y;
            m0z = z;
        } else {
            if (k == 1) {   // state at the first hit with the velocity of the first step
                abg_init(fy, m0y, y, d);
                abg_init(fz, m0z, z, d);
            }
            for (int j = 0; j < d; j++) {
                abg_predict(fy);
                abg_predict(fz);
            }
            abg_update(fy, y);
            abg_update(fz, z);
        }
        k++;
    }
};

constexpr int FO_CTAS = 10;      // blocks a multiprocessor: 48 registers a thread

// Each warp takes 32 x chunk tasks at a time from the queue (no CTA barrier: a warp whose chains
// end early takes the next ones while the others still follow theirs).  Task groups of 32 come in
// pairs: the outward tasks of 32 chains, then their inward tasks.  SKIP: chains may skip a row (the
// skip-row rule); the plain instantiation keeps the plain reading's registers.
template <bool SKIP, class T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? FO_CTAS : 1) k_follow(Work W, const int32_t *perm) {
    const DevGeom &g = *W.geom;
    const int nr = g.n_rows;
    const int lane = threadIdx.x & 31;
    int n_chains = W.counters[CNT_NCHAINS];
    if (n_chains > W.cap_chains) n_chains = W.cap_chains;
    const int n_groups = 2 * ((n_chains + 31) / 32);
    const int chunk = W.tune.chunk[3] > 0 ? W.tune.chunk[3] : 1;
    int32_t *q = W.counters + CNT_Q0 + 3;
    for (;;) {
        int base = 0;
        if (lane == 0) base = atomicAdd(q, chunk);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (base >= n_groups) break;
        for (int gr = base; gr < base + chunk && gr < n_groups; gr++) {
            const int i = (gr >> 1) * 32 + lane;
            if (i >= n_chains) continue;
            const int t = perm[i];
            const bool out = (gr & 1) == 0;
            const int len = W.chain_len[t], bin = W.chain_bin[t];
            const int row0 = bin % nr;
            const int rowbase = bin - row0;
            int32_t *slots = W.cand_slots + (size_t)t * nr;
            ChainFilter<T> f;
            int z_last = 0;
            const int dir = out ? 1 : -1;
            int x = out ? W.chain_start[t] : W.chain_last[t];
            const int32_t *link = out ? W.up : W.down;
            int row = out ? row0 : row0 + len - 1;
            if (SKIP && !out) {      // rows may be skipped: the last hit's row from its cluster
                int hi = nr - 1;
                while (row < hi) {
                    const int mid = (row + hi + 1) >> 1;
                    if (__ldg(W.bin_off + rowbase + mid) <= x) row = mid; else hi = mid - 1;
                }
            }
            int d = 1;
            for (int k = 0; k < len; k++) {
                const int y = __ldg(W.pad + x), z = __ldg(W.tim + x);
                const int nx = k + 1 < len ? __ldg(link + x) : 0;      // in flight with the coordinates
                if (out) slots[row] = x;
                f.hit(y, z, d);
                z_last = z;
                if (k + 1 < len) {
                    x = nx;
                    if constexpr (SKIP) {
                        // the next hit is one row on, or two across a row the link skips
                        if (out) {
                            d = row + 2 < nr && x >= __ldg(W.bin_off + rowbase + row + 2) ? 2 : 1;
                            if (d == 2) slots[row + 1] = -1;
                        } else {
                            d = row >= 1 && x < __ldg(W.bin_off + rowbase + row - 1) ? 2 : 1;
                        }
                    }
                    row += dir * d;
                }
            }
            int r_end = row;
            const bool far = sizeof(T) == 4 && z_last > NARROW_ZHIT;      // stops at its first row
            const int n = far ? 0 : extend(W, g, f.fy, f.fz, rowbase, row, dir, nr, slots, &r_end);
            // both threads of the chain add their part to the candidate (len hits and no rows so far)
            atomicAdd(W.cand_n + t, n);
            atomicAdd(W.cand_rows + t, out ? r_end << 16 : r_end);
        }
    }
}

// ---- few chains: eight lanes a task ----------------------------------------------------------------
// With few chains a step's latency is all that counts, and a thread alone pays for every dependent
// load of its search.  Here eight lanes share a task (one direction of a chain): they expand the
// chain together along its 1-, 2- and 4-link successors, carry the same filter state, and read a
// row's slabs 32 entries at a time, four per lane, without a search; the slab offsets of the next
// row are loaded during a row.  Same integer decisions as above; 32-bit filter, plain reading, at
// most FG_ROWS rows.
constexpr int FG = 8, FG_ROWS = 160, FG_BLOCK = 128, FG_CLUSTERS = 1 << 20;
__global__ void __launch_bounds__(FG_BLOCK) k_follow_few(Work W, const int32_t *perm, const int32_t *n1,
                                                         const int32_t *n2, const int32_t *n4) {
    __shared__ int32_t s_yz[FG_BLOCK / FG][FG_ROWS];      // the chain's coordinates, ascending rows
    using A = Abg<int>;
    constexpr unsigned FULL = 0xffffffffu;
    const DevGeom &g = *W.geom;
    const int nr = g.n_rows;
    const int lane = threadIdx.x & 31, j = lane & (FG - 1);
    const unsigned gmask = 0xffu << (lane & ~(FG - 1));
    int32_t *yzs = s_yz[threadIdx.x / FG];
    int n_chains = W.counters[CNT_NCHAINS];
    if (n_chains > W.cap_chains) n_chains = W.cap_chains;
    int32_t *q = W.counters + CNT_Q0 + 3;
    for (;;) {
        int base = 0;
        if (lane == 0) base = atomicAdd(q, 32 / FG);
        base = __shfl_sync(FULL, base, 0);
        if (base >= 2 * n_chains) break;
        const int task = base + lane / FG;
        const bool on = task < 2 * n_chains;
        const int t = on ? perm[task >> 1] : 0;
        const bool out = (task & 1) == 0;
        const int dir = out ? 1 : -1;
        const int len = on ? W.chain_len[t] : 0, bin = on ? W.chain_bin[t] : 0;
        const int row0 = bin % nr, rowbase = bin - row0;
        int32_t *slots = W.cand_slots + (size_t)t * nr;
        // lane j takes hits j, j + 8, ... of the chain
        int x = on ? W.chain_start[t] : 0;
        if (j < len) {
            if (j & 1) x = n1[x];
            if (j & 2) x = n2[x];
            if (j & 4) x = n4[x];
        }
        int rounds = len;
#pragma unroll
        for (int o = 16; o >= FG; o >>= 1) rounds = max(rounds, __shfl_xor_sync(FULL, rounds, o));
        for (int k = j; k - j < rounds; k += FG) {
            if (k < len) {
                const int y = __ldg(W.pad + x), z = __ldg(W.tim + x), c = x;
                if (k + FG < len) x = n4[n4[x]];
                yzs[k] = (int)((uint32_t)(y & 0xffff) | ((uint32_t)z << 16));
                if (out) slots[row0 + k] = c;
            }
        }
        __syncwarp();
        ChainFilter<int> f;
        f.fy = f.fz = A{0, 0, 0};
        int z_last = 0;
        for (int k = 0; k < rounds; k++) {
            if (k < len) {
                const int32_t v = yzs[out ? k : len - 1 - k];
                z_last = (int)((uint32_t)v >> 16);
                f.hit((int16_t)(v & 0xffff), z_last, 1);
            }
        }
        __syncwarp();
        // extension: every lane of the group holds the same state
        const int row_last = out ? row0 + len - 1 : row0;
        int row = row_last + dir, r_end = row_last, n = 0, misses = 0;
        int pend = -1, pend_row = -1;                        // this lane's found cluster, not stored yet
        bool act = on && z_last <= NARROW_ZHIT && row >= 0 && row < nr;
        // the coming row's cluster offset, and slab offsets zs .. zs + 7 of it (lane j holds zs + j)
        int c_next = 0, zs = 0, zo = 0;
        auto ahead = [&](int r, int pz) {
            zs = max(slab_of(max(pz - W_F0, 0)) - 2, 0);
            c_next = __ldg(W.bin_off + rowbase + r);
            zo = __ldg(W.zoff + (size_t)(rowbase + r) * ZOFF_STRIDE + min(zs + j, NZB));
        };
        if (act) ahead(row, q16_round(abg_ahead(f.fz)) + A::ZB);
        while (__any_sync(FULL, act)) {
            const int c0 = c_next, zs0 = zs, zo0 = zo;
            int py = 0, pz = 0, w = 0;
            if (act) {
                abg_predict(f.fy);
                abg_predict(f.fz);
                py = q16_round(f.fy.p);
                pz = q16_round(f.fz.p) + A::ZB;
                w = W_F0 + W_F1 * misses;
                if (abs(py) > g.ymax[row] || pz < 0 || pz > g.zmax || f.fy.v > V_MAX * 65536 || f.fy.v < -V_MAX * 65536)
                    act = false;
            }
            const int bin_r = rowbase + row;
            const int ps = act ? pstart_of(c0, bin_r) : 0;
            const int zl = slab_of(max(pz - w, 0)), zh = slab_of(pz + w);
            int lo = __shfl_sync(FULL, zo0, zl - zs0, FG), hi = __shfl_sync(FULL, zo0, zh + 1 - zs0, FG);
            if (act && (zl < zs0 || zh + 1 > zs0 + FG - 1)) {      // outside the offsets loaded ahead
                const uint16_t *zp = W.zoff + (size_t)bin_r * ZOFF_STRIDE;
                lo = __ldg(zp + zl);
                hi = __ldg(zp + zh + 1);
            }
            if (!act) lo = hi = 0;
            uint32_t bd = 0xffffffffu;          // this lane's smallest d^2, its position and payload
            int bi = 0, cnt = 0;
            int32_t bv = 0;
            bool first = true;
            for (int i0 = lo & ~3; __any_sync(FULL, i0 < hi); i0 += 4 * FG) {
                const int i = i0 + 4 * j;
                int4 e = make_int4(0, 0, 0, 0);
                if (i < hi) e = __ldg(reinterpret_cast<const int4 *>(W.gyz + ps + i));
                if (first) {                     // the next row's offsets, behind this row's entries
                    first = false;
                    if (act && row + dir >= 0 && row + dir < nr) ahead(row + dir, pz + (f.fz.v >> 16));
                    if (pend_row >= 0) slots[pend_row] = pend;
                    pend_row = -1;
                }
                const int32_t v[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
                for (int m = 0; m < 4; m++) {
                    const int dy = grid_y(v[m]) - py, dz = grid_z(v[m]) - pz;
                    if (i + m >= lo && i + m < hi && abs(dy) <= w && abs(dz) <= w) {
                        const uint32_t d2 = (uint32_t)(dy * dy + dz * dz);
                        if (d2 < bd) {
                            bd = d2;
                            bi = i + m;
                            bv = v[m];
                            cnt = 0;
                        }
                        cnt += d2 == bd;
                    }
                }
            }
            if (first) {                         // no entry in any group's slabs
                if (act && row + dir >= 0 && row + dir < nr) ahead(row + dir, pz + (f.fz.v >> 16));
                if (pend_row >= 0) slots[pend_row] = pend;
                pend_row = -1;
            }
            uint32_t m = bd;
#pragma unroll
            for (int o = FG / 2; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(FULL, m, o));
            const bool found = act && m <= (uint32_t)(w * w);
            bool mine = found && bd == m;
            const unsigned own = __ballot_sync(FULL, mine) & gmask, twice = __ballot_sync(FULL, mine && cnt > 1) & gmask;
            const bool tie = found && (__popc(own) > 1 || twice);
            if (__any_sync(FULL, tie)) {         // equal distances: the smallest index counts
                int bl = 0x7fffffff;
                if (tie && mine) {
                    for (int i0 = lo & ~3; i0 < hi; i0 += 4 * FG)
                        for (int i = i0 + 4 * j; i < min(i0 + 4 * j + 4, hi); i++) {
                            if (i < lo) continue;
                            const int32_t v = W.gyz[ps + i];
                            const int dy = grid_y(v) - py, dz = grid_z(v) - pz;
                            if (abs(dy) > w || abs(dz) > w || (uint32_t)(dy * dy + dz * dz) != m) continue;
                            const int l = W.gloc[ps + i];
                            if (l < bl) { bl = l; bi = i; bv = v; }
                        }
                }
                int ml = bl;
#pragma unroll
                for (int o = FG / 2; o > 0; o >>= 1) ml = min(ml, __shfl_xor_sync(FULL, ml, o));
                if (tie) mine = mine && bl == ml;
            }
            const unsigned who = __ballot_sync(FULL, mine) & gmask;
            const int32_t v = __shfl_sync(FULL, bv, who ? __ffs(who) - 1 : lane);
            if (act) {
                if (found) {
                    if (mine) {
                        pend = c0 + (int)__ldg(W.gloc + ps + bi);
                        pend_row = row;
                    }
                    abg_update(f.fy, grid_y(v));
                    abg_update(f.fz, grid_z(v) - A::ZB);
                    r_end = row;
                    n++;
                    misses = 0;
                } else {
                    if (j == 0) slots[row] = -1;
                    if (++misses >= M_MISS) act = false;
                }
                row += dir;
                if (row < 0 || row >= nr) act = false;
            }
        }
        if (pend_row >= 0) slots[pend_row] = pend;
        if (on && j == 0) {
            atomicAdd(W.cand_n + t, n);
            atomicAdd(W.cand_rows + t, out ? r_end << 16 : r_end);
        }
        __syncwarp();
    }
}

}  // namespace

int follow_narrow(const DevGeom &g) { return g.ymax[g.n_rows - 1] <= NARROW_YMAX && g.zmax <= NARROW_ZMAX; }

void launch_follow(const Work &W, cudaStream_t s) {
    const int block = W.tune.block[3] > 0 ? W.tune.block[3] : 128;
    const int grid = W.tune.grid[3] > 0 ? W.tune.grid[3] : W.sm_count * FO_CTAS;
    int32_t *perm = W.perm;
    k_follow_order<<<W.sm_count * 8, 256, 0, s>>>(W, perm);
    // Few chains (about one per 30 clusters): eight lanes a task.  Measured, a thread / eight lanes a
    // task: one sector (138 chains) 214 / 136 us, 5,000-track event (17,885 chains of 0.92 M clusters)
    // 317 / 283, 12 events (35,942 of 2.3 M) 327 / 345, central event (135,775 of 3.9 M) 651 / 2021.
    if (W.narrow && !(W.rules & TPC_RULE_SKIP_ROW) && W.nr <= FG_ROWS && W.n_clusters <= FG_CLUSTERS) {
        // the successors are those of the chain stage (still there: the selection overwrites two)
        const int32_t *n1 = reinterpret_cast<const int32_t *>(W.claim);
        k_follow_few<<<W.sm_count * 12, FG_BLOCK, 0, s>>>(W, perm, n1, n1 + (W.n_clusters + 1), W.jump4);
        return;
    }
    if (W.rules & TPC_RULE_SKIP_ROW)
        W.narrow ? k_follow<true, int><<<grid, block, 0, s>>>(W, perm)
                 : k_follow<true, long long><<<grid, block, 0, s>>>(W, perm);
    else
        W.narrow ? k_follow<false, int><<<grid, block, 0, s>>>(W, perm)
                 : k_follow<false, long long><<<grid, block, 0, s>>>(W, perm);
}

}  // namespace tpc
