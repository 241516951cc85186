// S7 inter-sector merging (arxiv 1712.09434 section 3: sectors are tracked independently and
// concurrently, and the track segments are merged afterwards) and assembly of the output tracks.
//
// Ends: the first kept hit of a segment, and its outer end = last kept hit plus the kept hit
// MERGE_BACK positions earlier, on integer (Xtab[row], Y, Z).  The outer end of S is rotated into
// an adjacent sector of the same side with Q30 integer constants (floor shifts), extrapolated
// linearly (floor division) to the row of T's first hit and compared there.  Every valid pair
// offers (D, index) to both sides with 64-bit atomicMin; mutual bests are linked S -> T.  A chain
// of links is one track; a cycle is cut in front of its smallest segment.  Track ids are an
// exclusive scan of head flags in segment order (= seed order), so the output order is canonical.
#include "tpc_common.cuh"

namespace tpc {

namespace {

__device__ __forceinline__ int n_chains_of(const Work &W) {
    const int n = W.counters[CNT_NCHAINS];
    return n < W.cap_chains ? n : W.cap_chains;
}

// Kept hits of an accepted candidate: a bit per row of its row range [r0, r1], from r0 on.
struct Kept {
    const uint32_t *w;
    int r0, r1;
    __device__ __forceinline__ bool has(int r) const { return (w[(r - r0) >> 5] >> ((r - r0) & 31)) & 1u; }
    // row of the first kept hit
    __device__ __forceinline__ int first() const {
        for (int j = 0; j <= (r1 - r0) >> 5; j++)
            if (w[j]) return r0 + 32 * j + __ffs(w[j]) - 1;
        return -1;
    }
    // row of the last kept hit and of the kept hit `back` positions before it (-1 if there is none)
    __device__ __forceinline__ void last(int back, int &rl, int &rb) const {
        rl = rb = -1;
        for (int j = (r1 - r0) >> 5; j >= 0; j--) {
            uint32_t m = w[j];
            while (m) {
                const int bit = 31 - __clz(m), r = r0 + 32 * j + bit;
                if (rl < 0) rl = r;
                if (back-- == 0) { rb = r; return; }
                m &= ~(1u << bit);
            }
        }
    }
};
__device__ __forceinline__ Kept kept_of(const Work &W, int t) {
    const int rr = W.cand_rows[t];
    return Kept{W.kept + (size_t)t * kept_words(W.nr), rr & 0xffff, rr >> 16};
}

// ends of accepted segments; reset of the merge arrays
__global__ void k_merge_ends(Work W) {
    const DevGeom &g = *W.geom;
    const int n = n_chains_of(W);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        W.bestT[t] = ~0ull;
        W.bestS[t] = ~0ull;
        W.next[t] = -1;
        W.prev[t] = -1;
        if (W.seg_n[t] < N_MIN) continue;
        const Kept kept = kept_of(W, t);
        const int32_t *sl = W.cand_slots + (size_t)t * W.nr;
        const int rf = kept.first();
        int rL, rB;
        kept.last(MERGE_BACK, rL, rB);
        if (rB < 0) { set_status(W, ST_BOUNDS); continue; }
        const int first = sl[rf], hL = sl[rL], hB = sl[rB];
        const int sector = (W.chain_bin[t] % (W.ns * W.nr)) / W.nr;
        W.inend[t] = make_int4(g.xtab[rf], W.pad[first], W.tim[first], sector);
        atomicMax(W.sec_ymax + W.chain_bin[t] / (W.ns * W.nr) * W.ns + sector, abs((int)W.pad[first]));
        atomicAdd(W.bin_cnt + (W.chain_bin[t] - W.chain_bin[t] % W.nr) + rf, 1);
        W.outend[2 * t] = make_int4(g.xtab[rB], W.pad[hB], W.tim[hB], sector);
        W.outend[2 * t + 1] = make_int4(g.xtab[rL], W.pad[hL], W.tim[hL], rL);
    }
}

// Accepted segments listed per (event, sector, row of the first kept hit): the merge only looks at
// segments whose first row lies inside the extrapolation reach, and reads their first hits (Xtab, Y,
// Z, index) in that order.
__device__ __forceinline__ int4 *merge_firsts(const Work &W) {
    // behind the list of outer ends, in the packed track hits (written later)
    return reinterpret_cast<int4 *>(W.trk_pack + ((2 * (size_t)W.cap_chains + 3) & ~(size_t)3));
}
__global__ void k_merge_fill(Work W) {
    const int n = n_chains_of(W);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
        if (W.seg_n[t] < N_MIN) continue;
        const int4 e = W.inend[t];
        const int bin0 = W.chain_bin[t] - W.chain_bin[t] % W.nr;
        int lo = 0, hi = W.nr - 1;   // row of the first kept hit from its Xtab value
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (W.geom->xtab[mid] < e.x) lo = mid + 1; else hi = mid;
        }
        const int b = bin0 + lo;
        const int p = W.mrg_off[b] + atomicSub(W.bin_cnt + b, 1) - 1;
        merge_firsts(W)[p] = make_int4(e.x, e.y, e.z, t);
    }
}

// ---- gap merge inside a sector (TPC_RULE_GAP_MERGE) --------------------------------------------
// The integer steady-state filter of the following (alpha-beta-gamma 1/2, 1/8, 1/32, Q16, floor
// shifts) runs over the kept hits of a segment, one step per pad row and an update per kept hit.
struct Abg {
    long long p, v, a;
};
__device__ __forceinline__ void abg_init(Abg &f, long long m0, long long m1, long long drow) {
    f.p = m0 * 65536;
    f.v = floor_div((m1 - m0) * 65536, drow);
    f.a = 0;
}
__device__ __forceinline__ void abg_predict(Abg &f) {
    f.p += f.v + (f.a >> 1);
    f.v += f.a;
}
__device__ __forceinline__ void abg_update(Abg &f, long long m) {
    const long long e = m * 65536 - f.p;
    f.p += e >> 1;
    f.v += e >> 3;
    f.a += e >> 5;
}
__device__ __forceinline__ long long q16_round(long long p) { return (p + 32768) >> 16; }
__device__ __forceinline__ bool gap_inside(const DevGeom &g, const Abg &fy, const Abg &fz, int row) {
    const long long py = q16_round(fy.p), pz = q16_round(fz.p);
    const long long av = fy.v < 0 ? -fy.v : fy.v;
    return !((py < 0 ? -py : py) > g.ymax[row] || pz < 0 || pz > g.zmax || av > (long long)V_MAX * 65536);
}

// Calls f(row, y, z) for the kept hits of a segment in ascending (DIR +1) or descending rows; the
// hits are loaded four at a time.
template <int DIR, class F>
__device__ __forceinline__ void kept_walk(const Work &W, const Kept &kept, const int32_t *sl, F f) {
    const int last = (kept.r1 - kept.r0) >> 5;
    int j = DIR > 0 ? 0 : last;
    uint32_t m = kept.w[j];
    for (;;) {
        int row[4], h[4], y[4], z[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            while (!m && j + DIR >= 0 && j + DIR <= last) {
                j += DIR;
                m = kept.w[j];
            }
            row[q] = -1;
            if (m) {
                const int bit = DIR > 0 ? __ffs(m) - 1 : 31 - __clz(m);
                row[q] = kept.r0 + 32 * j + bit;
                m &= ~(1u << bit);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; q++) h[q] = row[q] >= 0 ? sl[row[q]] : 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            y[q] = row[q] >= 0 ? W.pad[h[q]] : 0;
            z[q] = row[q] >= 0 ? W.tim[h[q]] : 0;
        }
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (row[q] >= 0) f(row[q], y[q], z[q]);
        if (row[3] < 0) return;
    }
}

// The filter over the kept hits of a segment in one direction; row, y0 and z0 are those of the last
// hit taken.
struct SegFilter {
    Abg fy{}, fz{};
    int k = 0, row = 0, y0 = 0, z0 = 0;
    __device__ __forceinline__ void hit(int r, int y, int z) {
        const int d = r > row ? r - row : row - r;
        if (k > 0) {
            if (k == 1) {
                abg_init(fy, y0, y, d);
                abg_init(fz, z0, z, d);
            }
            for (int j = d; j > 0; j--) {
                abg_predict(fy);
                abg_predict(fz);
            }
            abg_update(fy, y);
            abg_update(fz, z);
        }
        row = r;
        y0 = y;
        z0 = z;
        k++;
    }
};

// Accepted segments as a list in warp order (a fifth of the chains: the kernels below run with full
// warps on it), and the reset of the gap keys.
__global__ void __launch_bounds__(128) k_gap_list(Work W, int32_t *list) {
    const int n = n_chains_of(W);
    const int lane = threadIdx.x & 31;
    for (int t0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); t0 < n; t0 += gridDim.x * blockDim.x) {
        const int t = t0 + lane;
        bool acc = false;
        if (t < n) {
            W.gap_bestT[t] = ~0ull;
            W.gap_bestS[t] = ~0ull;
            acc = W.seg_n[t] >= N_MIN;
        }
        const unsigned m = __ballot_sync(0xffffffffu, acc);
        int p = 0;
        if (lane == 0 && m) p = atomicAdd(W.counters + CNT_GAP, __popc(m));
        p = __shfl_sync(0xffffffffu, p, 0);
        if (acc) list[p + __popc(m & ((1u << lane) - 1u))] = t;
    }
}

// Forward filter state of a segment at its last kept hit: five words in the selection's claims (five
// clusters or more per chain), the sixth in the 4-link successors; both are free by now.
__device__ __forceinline__ long long *gap_fwd(const Work &W, int t, int k) {
    return k < 5 ? reinterpret_cast<long long *>(W.claim) + 5 * (size_t)t + k
                 : reinterpret_cast<long long *>(W.jump4) + t;
}

// Both filters of every accepted segment over its kept hits, a thread each: in descending rows to the
// state at its first kept hit, and in ascending rows to the state at its last.
__global__ void __launch_bounds__(128) k_gap_filter(Work W, const int32_t *list) {
    const int n = W.counters[CNT_GAP];
    const int n32 = (n + 31) & ~31;           // warps of one direction
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * n32; i += gridDim.x * blockDim.x) {
        const bool back = i < n32;
        const int q = back ? i : i - n32;
        if (q >= n) continue;
        const int t = list[q];
        const Kept kept = kept_of(W, t);
        const int32_t *sl = W.cand_slots + (size_t)t * W.nr;
        SegFilter f;
        if (back) kept_walk<-1>(W, kept, sl, [&](int r, int y, int z) { f.hit(r, y, z); });
        else kept_walk<1>(W, kept, sl, [&](int r, int y, int z) { f.hit(r, y, z); });
        const long long st[6] = {f.fy.p, f.fy.v, f.fy.a, f.fz.p, f.fz.v, f.fz.a};
#pragma unroll
        for (int k = 0; k < 6; k++) *(back ? W.gap_state + 6 * (size_t)t + k : gap_fwd(W, t, k)) = st[k];
    }
}

// Warp per segment S: its forward filter row by row across the gap; the lanes test the segments T of
// the same sector whose first kept hit lies k >= M_MISS + 1 rows past S's last kept hit, both ways;
// (D, T) kept for S, (D, S) offered to T by 64-bit atomicMin.  Behind a range of dead rows hundreds
// of segments start in one row, and a thread per S took them one after the other: 79 + 333 us for
// both filters and the tests of 147 k chains (28,991 tracks), now 5 + 74 + 134.
__global__ void __launch_bounds__(128) k_gap_match(Work W, const int32_t *list) {
    const DevGeom &g = *W.geom;
    const int n = W.counters[CNT_GAP];
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int i0 = gw; i0 < n; i0 += nw) {
        const int s = list[i0];
        Abg fy{*gap_fwd(W, s, 0), *gap_fwd(W, s, 1), *gap_fwd(W, s, 2)};
        Abg fz{*gap_fwd(W, s, 3), *gap_fwd(W, s, 4), *gap_fwd(W, s, 5)};
        const int4 last = W.outend[2 * s + 1];
        const int rs = last.w;
        const long long ys = last.y, zs = last.z;
        const int b0 = W.chain_bin[s] - W.chain_bin[s] % W.nr;   // (event, sector) row 0
        unsigned long long best = ~0ull;
        for (int rt = rs + 1; rt < W.nr && rt <= rs + GAP_MAX; rt++) {
            abg_predict(fy);
            abg_predict(fz);
            if (!gap_inside(g, fy, fz, rt)) break;
            if (rt - rs - 1 < M_MISS) continue;
            const long long py = q16_round(fy.p), pz = q16_round(fz.p);
            const long long w = W_F0 + (long long)W_F1 * (rt - rs - 1);
            const int i1 = W.mrg_off[b0 + rt + 1];
            for (int i = W.mrg_off[b0 + rt] + lane; i < i1; i += 32) {
                const int4 e = merge_firsts(W)[i];
                const int t = e.w;
                if (t == s) continue;
                const long long dy = e.y - py, dz = e.z - pz;
                if (dy > w || dy < -w || dz > w || dz < -w || dy * dy + dz * dz > w * w) continue;
                const long long *st = W.gap_state + 6 * (size_t)t;
                Abg by{st[0], st[1], st[2]}, bz{st[3], st[4], st[5]};
                bool inside = true;
                for (int j = 1; j <= rt - rs && inside; j++) {
                    abg_predict(by);
                    abg_predict(bz);
                    inside = gap_inside(g, by, bz, rt - j);
                }
                if (!inside) continue;
                const long long ey = ys - q16_round(by.p), ez = zs - q16_round(bz.p);
                if (ey > w || ey < -w || ez > w || ez < -w || ey * ey + ez * ez > w * w) continue;
                const unsigned long long D = (unsigned long long)(dy * dy + dz * dz + ey * ey + ez * ez);
                const unsigned long long kT = (D << 32) | (unsigned)t;
                best = kT < best ? kT : best;
                atomicMin(W.gap_bestS + t, (D << 32) | (unsigned)s);
            }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, d);
            best = v < best ? v : best;
        }
        if (lane == 0) W.gap_bestT[s] = best;
    }
}

// Mutual best gap pairs become merge links S -> T before the sector merge runs.
__global__ void k_gap_link(Work W) {
    const int n = n_chains_of(W);
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        const unsigned long long v = W.gap_bestT[s];
        if (v == ~0ull) continue;
        const int t = (int)(v & 0xffffffffu);
        if (W.gap_bestS[t] == ((v & 0xffffffff00000000ull) | (unsigned)s)) {
            W.next[s] = t;
            W.prev[t] = s;
        }
    }
}

// The outer end of segment S in the frame of the adjacent sector on side k (0: the next, 1: the
// previous one).
struct OuterEnd {
    long long x1, y1, x2, y2, dxs;
    int z1, dz, kt;        // Z of the inner point, Z difference, sector
};
__device__ __forceinline__ bool outer_end(const Work &W, const DevGeom &g, int s, int k, OuterEnd &o) {
    const int half = W.ns / 2;
    const int4 p1 = W.outend[2 * s], p2 = W.outend[2 * s + 1];
    const int ks = p1.w;
    const int side0 = ks < half ? 0 : half;
    const int sgn = k == 0 ? +1 : -1;
    o.kt = side0 + ((ks - side0) + (k == 0 ? 1 : half - 1)) % half;
    if (k == 1 && o.kt == side0 + ((ks - side0) + 1) % half) return false;   // tiny geometries
    const long long X1 = p1.x, Y1 = p1.y, X2 = p2.x, Y2 = p2.y;
    o.x1 = (X1 * g.c30 + sgn * Y1 * g.s30) >> 30;
    o.y1 = (-sgn * X1 * g.s30 + Y1 * g.c30) >> 30;
    o.x2 = (X2 * g.c30 + sgn * Y2 * g.s30) >> 30;
    o.y2 = (-sgn * X2 * g.s30 + Y2 * g.c30) >> 30;
    o.dxs = o.x2 - o.x1;
    o.z1 = p1.z;
    o.dz = p2.z - p1.z;
    return o.dxs > 0;
}

// Thread per (outer end, adjacent sector): lists those that can match anything.  The extrapolated Y
// is monotonic in XT, so its range over the reach |XT - x2| <= MERGE_XMAX is that of the two ends.
// If the window around it misses the range of the first-hit Y of every segment of that sector, no T
// there can match (the usual case: S ends away from the edge that faces it).  This decision is the
// same for all T, so it is taken with full warps here and not by each lane of the warps that match.
// With the first hits read in bucket order and tested in FP32 before the 64-bit arithmetic, both
// kernels take 494 us on 64 events (923 as one), 67 us on a central event (170).
__global__ void __launch_bounds__(128) k_merge_probe(Work W, int32_t *list) {
    const DevGeom &g = *W.geom;
    const long long n2 = 2ll * n_chains_of(W);
    const int lane = threadIdx.x & 31;
    const bool gap = (W.rules & TPC_RULE_GAP_MERGE) != 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n2; i0 += stride) {
        const long long i = i0 + lane;
        const int s = (int)(i >> 1), k = (int)(i & 1);
        bool keep = false;
        if (i < n2 && W.seg_n[s] >= N_MIN && !(gap && W.next[s] >= 0)) {    // a gap successor: no outer end
            OuterEnd o;
            if (outer_end(W, g, s, k, o)) {
                const long long ya = o.y1 + floor_div_pos((o.x2 - MERGE_XMAX - o.x1) * (o.y2 - o.y1), o.dxs);
                const long long yb = o.y1 + floor_div_pos((o.x2 + MERGE_XMAX - o.x1) * (o.y2 - o.y1), o.dxs);
                const long long ymin = ya < yb ? ya : yb, ymx = ya < yb ? yb : ya;
                const long long bound = W.sec_ymax[W.chain_bin[s] / (W.ns * W.nr) * W.ns + o.kt];
                keep = !(ymin - W_MERGE > bound || ymx + W_MERGE < -bound);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (!m) continue;
        int p = 0;
        if (lane == 0) p = atomicAdd(W.counters + CNT_MERGE, __popc(m));
        p = __shfl_sync(0xffffffffu, p, 0);
        if (keep) list[p + __popc(m & ((1u << lane) - 1u))] = (int32_t)((uint32_t)s << 1 | (uint32_t)k);
    }
}

// One warp per listed outer end S and adjacent sector: the lanes take the candidate segments T of the
// reachable rows 32 at a time; every valid pair offers (D, T) to S and (D, S) to T with 64-bit
// atomicMin (for S once per warp).
__global__ void __launch_bounds__(128) k_merge_match(Work W, const int32_t *list) {
    const DevGeom &g = *W.geom;
    const int n = W.counters[CNT_MERGE];
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    const float pitch = (float)(g.xtab[W.nr - 1] - g.xtab[0]) / (float)(W.nr - 1);
    const bool gap = (W.rules & TPC_RULE_GAP_MERGE) != 0;
    for (int q = gw; q < n; q += nw) {
        const int s = (int)((uint32_t)list[q] >> 1);
        OuterEnd o;
        outer_end(W, g, s, list[q] & 1, o);
        const int b0 = (W.chain_bin[s] / (W.ns * W.nr) * W.ns + o.kt) * W.nr;
        // rows whose plane is within MERGE_XMAX of the extrapolation start (one row of margin; the exact
        // test is below)
        int r_lo = (int)floorf((float)(o.x2 - MERGE_XMAX - g.xtab[0]) / pitch) - 1;
        int r_hi = (int)ceilf((float)(o.x2 + MERGE_XMAX - g.xtab[0]) / pitch) + 1;
        r_lo = max(r_lo, 0);
        r_hi = min(r_hi, W.nr - 1);
        if (r_lo > r_hi) continue;
        unsigned long long best = ~0ull;
        const float fy = (float)(o.y2 - o.y1) / (float)o.dxs, fz = (float)o.dz / (float)o.dxs;
        const float y1 = (float)o.y1, z1 = (float)o.z1;
        const int i1 = W.mrg_off[b0 + r_hi + 1];
        for (int i = W.mrg_off[b0 + r_lo] + lane; i < i1; i += 32) {
            const int4 e = merge_firsts(W)[i];
            const long long XT = e.x;
            const long long ax = XT - o.x2;
            if ((ax < 0 ? -ax : ax) > MERGE_XMAX) continue;
            {   // the windows in FP32, with margins above the floor and the rounding (a few 2^-24 of the
                // terms): only pairs that the integer tests below reject are dropped
                const float dx = (float)(XT - o.x1), py = dx * fy, pz = dx * fz;
                if (fabsf((float)e.y - y1 - py) > (float)W_MERGE + 2.f + 1e-6f * (fabsf(y1) + fabsf(py)) ||
                    fabsf((float)e.z - z1 - pz) > (float)W_MERGE + 2.f + 1e-6f * (fabsf(z1) + fabsf(pz)))
                    continue;
            }
            const int t = e.w;
            if (gap && W.prev[t] >= 0) continue;                 // a gap predecessor: no first segment
            const long long yp = o.y1 + floor_div_pos((XT - o.x1) * (o.y2 - o.y1), o.dxs);
            const long long zp = o.z1 + floor_div_pos((XT - o.x1) * (long long)o.dz, o.dxs);
            const long long dy = e.y - yp, dz = e.z - zp;
            if (dy > W_MERGE || dy < -W_MERGE || dz > W_MERGE || dz < -W_MERGE) continue;
            const unsigned long long D = (unsigned long long)(dy * dy + dz * dz);
            const unsigned long long kT = (D << 32) | (unsigned)t;
            best = kT < best ? kT : best;
            atomicMin(W.bestS + t, (D << 32) | (unsigned)s);
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, d);
            best = v < best ? v : best;
        }
        if (lane == 0 && best != ~0ull) atomicMin(W.bestT + s, best);
    }
}

__global__ void k_merge_link(Work W) {
    const int n = n_chains_of(W);
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        const unsigned long long v = W.bestT[s];
        if (v == ~0ull) continue;
        const int t = (int)(v & 0xffffffffu);
        if (W.bestS[t] == ((v & 0xffffffff00000000ull) | (unsigned)s)) {
            W.next[s] = t;
            W.prev[t] = s;
        }
    }
}

__global__ void k_merge_heads(Work W) {
    const int n = n_chains_of(W);
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        int head = 0;
        if (W.seg_n[s] >= N_MIN) {
            if (W.prev[s] < 0) {
                head = 1;
            } else {
                int x = W.prev[s], k = 0;
                while (x >= 0 && x != s && k < MERGE_MAX_WALK) { x = W.prev[x]; k++; }
                if (k >= MERGE_MAX_WALK) {
                    set_status(W, ST_TIMEOUT);
                } else if (x == s) {       // on a cycle: the smallest segment starts the track
                    int m = s, y = W.next[s];
                    k = 0;
                    while (y != s && k < MERGE_MAX_WALK) { m = y < m ? y : m; y = W.next[y]; k++; }
                    head = m == s;
                }
            }
        }
        W.head[s] = head;
    }
}

// hits per track (walk the segment chain from its head)
__global__ void k_track_count(Work W) {
    const int n = n_chains_of(W);
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        if (!W.head[s]) continue;
        const int tid = W.head_id[s];
        if (tid >= W.cap_tracks) { set_status(W, ST_CAPACITY); continue; }
        int sum = 0, x = s, k = 0;
        do {
            sum += W.seg_n[x];
            x = W.next[x];
            k++;
        } while (x >= 0 && !W.head[x] && k < MERGE_MAX_WALK);
        W.trk_n[tid] = sum;
        W.trk_head[tid] = s;
    }
}

// One warp per track: the lanes take the row slots of a segment 32 at a time, TW_ILP groups loaded
// together, and write its kept hits in row order (prefix of the kept bits), then move to the next
// segment of the merge chain.
constexpr int TW_ILP = 5;
__global__ void k_track_write(Work W) {
    const int nt = min(W.counters[CNT_NTRACKS], W.cap_tracks);
    const int lane = threadIdx.x & 31;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int tid = gw; tid < nt; tid += nw) {
        int pos = W.trk_off[tid];
        int x = W.trk_head[tid], k = 0;
        do {
            const Kept kept = kept_of(W, x);
            const int32_t *sl = W.cand_slots + (size_t)x * W.nr;
            const int sector = (W.chain_bin[x] % (W.ns * W.nr)) / W.nr;
            const int nwords = ((kept.r1 - kept.r0) >> 5) + 1;
            for (int j0 = 0; j0 < nwords; j0 += TW_ILP) {
                int h[TW_ILP], yz[TW_ILP];
                unsigned m[TW_ILP];
#pragma unroll
                for (int j = 0; j < TW_ILP; j++) {
                    m[j] = j0 + j < nwords ? kept.w[j0 + j] : 0u;
                    const int r = kept.r0 + 32 * (j0 + j) + lane;
                    h[j] = r <= kept.r1 ? sl[r] : -1;
                }
#pragma unroll
                for (int j = 0; j < TW_ILP; j++)
                    if ((m[j] >> lane) & 1u)
                        yz[j] = (int)((uint32_t)(W.pad[h[j]] & 0xffff) | ((uint32_t)W.tim[h[j]] << 16));
#pragma unroll
                for (int j = 0; j < TW_ILP; j++) {
                    if ((m[j] >> lane) & 1u) {
                        const int p = pos + __popc(m[j] & ((1u << lane) - 1u));
                        const int r = kept.r0 + 32 * (j0 + j) + lane;
                        if (p < W.cap_hits) {
                            W.trk_hits[p] = h[j];
                            W.label[h[j]] = tid;
                            reinterpret_cast<int2 *>(W.trk_pack)[p] = make_int2(yz[j], sector | (r << 16));
                        } else {
                            set_status(W, ST_CAPACITY);
                        }
                    }
                    pos += __popc(m[j]);
                }
            }
            x = W.next[x];
            k++;
        } while (x >= 0 && !W.head[x] && k < MERGE_MAX_WALK);
    }
}

__global__ void k_event_offsets(Work W) {
    const int n = n_chains_of(W);
    const int nbe = W.ns * W.nr;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e <= W.n_events; e += gridDim.x * blockDim.x) {
        if (e == W.n_events) {
            W.ev_trk_off[e] = W.counters[CNT_NTRACKS];
            *W.n_tracks = W.counters[CNT_NTRACKS];
        } else {
            W.ev_trk_off[e] = W.head_id[min(W.chain_off[e * nbe], n)];
        }
    }
}

}  // namespace

void launch_merge(const Work &W, cudaStream_t s) {
    const int block = W.tune.block[5] > 0 ? W.tune.block[5] : 128;
    const int grid = W.tune.grid[5] > 0 ? W.tune.grid[5] : W.sm_count * 8;
    // bin_cnt and sec_ymax were reset by the chain stage
    k_merge_ends<<<grid, block, 0, s>>>(W);
    scan_exclusive(W.bin_cnt, W.mrg_off, W.nbins, nullptr, nullptr, W.scan_tmp, W.scan_tmp_len, s);
    k_merge_fill<<<grid, block, 0, s>>>(W);
    if (W.rules & TPC_RULE_GAP_MERGE) {
        // the list lives in the track heads, which are written below
        k_gap_list<<<W.sm_count * 8, 128, 0, s>>>(W, W.trk_head);
        k_gap_filter<<<W.sm_count * 10, 128, 0, s>>>(W, W.trk_head);
        k_gap_match<<<W.sm_count * 14, 128, 0, s>>>(W, W.trk_head);
        k_gap_link<<<grid, block, 0, s>>>(W);
    }
    // the list lives in the packed track hits, which are written below
    k_merge_probe<<<W.sm_count * 8, 128, 0, s>>>(W, W.trk_pack);
    k_merge_match<<<W.sm_count * 12, 128, 0, s>>>(W, W.trk_pack);
    k_merge_link<<<grid, block, 0, s>>>(W);
    k_merge_heads<<<grid, block, 0, s>>>(W);
    scan_exclusive(W.head, W.head_id, W.cap_chains, W.counters + CNT_NCHAINS, W.counters + CNT_NTRACKS,
                   W.scan_tmp, W.scan_tmp_len, s);
    k_track_count<<<grid, block, 0, s>>>(W);
    scan_exclusive(W.trk_n, W.trk_off, W.cap_tracks, W.counters + CNT_NTRACKS, W.counters + CNT_NHITS,
                   W.scan_tmp, W.scan_tmp_len, s);
    k_track_write<<<grid, block, 0, s>>>(W);
    k_event_offsets<<<1, 128, 0, s>>>(W);
}

}  // namespace tpc
