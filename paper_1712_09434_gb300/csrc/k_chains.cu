// S3 link cleaning and S4 chains (seeds of the cellular automaton; arxiv 1712.09434 section 3:
// short track candidates of five to ten hits built from neighbour links).
//
// A link c -> u is kept only if it is mutual (down[u] == c); both directions read the uncleaned
// arrays.  The kept up-links are written once, with their 2- and 4-link successors (pointer
// jumping), so that a chain walk takes four links per dependent load.  A chain starts at a cluster
// with a kept up-link and no kept down-link and follows the kept up-links; chains of at least
// N_SEED hits are compacted in start-cluster order: per-bin counts (one warp per bin), a
// device-wide scan, and an ordered warp-ballot compaction.
//
// What bounds it: gathers into the neighbouring rows and the dependent loads of the walks.  One
// sweep reads both link arrays, decides links and starts and lists the starts (one cluster in
// twenty or thirty), so that the walks run with full warps, one start a lane, and the later passes
// read one word a cluster; every sweep has several clusters per thread in flight.  Measured, a
// sweep that also walked, warp per bin -> this (all passes): 64 events 1250 -> 775 us, central event
// 165 -> 77, 5,000-track event 120 -> 51, one sector 64 -> 30.
#include "tpc_common.cuh"

namespace tpc {

namespace {

// Kept up-link of every cluster (-1 if none or not mutual), and the successors 2 and 4 links
// further: a chain walk then takes four links per dependent load.  The first two live in the
// selection's claim words, which the selection re-initialises before use.
struct Jumps {
    int32_t *n1, *n2, *n4;
};
__device__ __forceinline__ Jumps jumps_of(const Work &W) {
    Jumps j;
    j.n1 = reinterpret_cast<int32_t *>(W.claim);
    j.n2 = reinterpret_cast<int32_t *>(W.claim) + (W.n_clusters + 1);
    j.n4 = W.jump4;
    return j;
}

// last cluster of the chain that starts at c, and the list of starts: in the packed track hits, which
// are written later
__device__ __forceinline__ int32_t *chain_ends(const Work &W) { return W.trk_pack; }
__device__ __forceinline__ int32_t *start_list(const Work &W) { return W.trk_pack + W.n_clusters; }

constexpr int SWEEP = 4;      // clusters per thread in flight

// Kept up-links, and the list of chain starts (in no particular order; every warp collects its starts
// in shared memory and appends them a hundred or so at a time, since one counter update per 32
// clusters alone took 0.5 ms on 64 events).
constexpr int START_BUF = 256;
__global__ void __launch_bounds__(256) k_mutual(Work W) {
    __shared__ int32_t s_buf[8][START_BUF];
    const Jumps J = jumps_of(W);
    const int lane = threadIdx.x & 31;
    int32_t *buf = s_buf[threadIdx.x >> 5];
    int n_buf = 0;                     // the same in all lanes
    const long long n = W.n_clusters, stride = (long long)gridDim.x * blockDim.x;
    auto flush = [&]() {
        int p = 0;
        if (lane == 0) p = atomicAdd(W.counters + CNT_STARTS, n_buf);
        p = __shfl_sync(0xffffffffu, p, 0);
        __syncwarp();
        for (int i = lane; i < n_buf; i += 32) start_list(W)[p + i] = buf[i];
        __syncwarp();
        n_buf = 0;
    };
    for (long long c0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); c0 < n; c0 += SWEEP * stride) {
        int u[SWEEP], d[SWEEP];
#pragma unroll
        for (int j = 0; j < SWEEP; j++) {
            const long long c = c0 + lane + j * stride;
            u[j] = c < n ? W.up[c] : -1;
            d[j] = c < n ? W.down[c] : -1;
        }
        int ud[SWEEP], du[SWEEP];
#pragma unroll
        for (int j = 0; j < SWEEP; j++) {
            ud[j] = u[j] >= 0 ? W.down[u[j]] : -1;
            du[j] = d[j] >= 0 ? W.up[d[j]] : -1;
        }
#pragma unroll
        for (int j = 0; j < SWEEP; j++) {
            const long long c = c0 + lane + j * stride;
            const bool kept = u[j] >= 0 && ud[j] == (int)c;
            const bool start = kept && !(d[j] >= 0 && du[j] == (int)c);
            if (c < n) {
                J.n1[c] = kept ? u[j] : -1;
                W.clen[c] = 0;
            }
            const unsigned m = __ballot_sync(0xffffffffu, start);
            if (start) buf[n_buf + __popc(m & ((1u << lane) - 1u))] = (int)c;
            n_buf += __popc(m);
        }
        if (n_buf > START_BUF - 32 * SWEEP) flush();
    }
    if (n_buf > 0) flush();
}

__global__ void __launch_bounds__(256) k_jump(Work W, const int32_t *src, int32_t *dst) {
    const long long n = W.n_clusters, stride = (long long)gridDim.x * blockDim.x;
    for (long long c0 = blockIdx.x * blockDim.x + threadIdx.x; c0 < n; c0 += SWEEP * stride) {
        int u[SWEEP], v[SWEEP];
#pragma unroll
        for (int j = 0; j < SWEEP; j++) u[j] = c0 + j * stride < n ? src[c0 + j * stride] : -1;
#pragma unroll
        for (int j = 0; j < SWEEP; j++) v[j] = u[j] >= 0 ? src[u[j]] : -1;
#pragma unroll
        for (int j = 0; j < SWEEP; j++)
            if (c0 + j * stride < n) dst[c0 + j * stride] = v[j];
    }
}

// Length and last cluster of the chain of every listed start (at most max_len hits).
__global__ void __launch_bounds__(128) k_chain_walk(Work W) {
    const Jumps J = jumps_of(W);
    const int n = W.counters[CNT_STARTS], max_len = W.geom->n_rows;
    const int32_t *list = start_list(W);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = list[i];
        int len = 1, x = c;
        while (len < max_len) {
            if (len + 4 <= max_len) {
                const int y = J.n4[x];
                if (y >= 0) { x = y; len += 4; continue; }
            }
            if (len + 2 <= max_len) {
                const int y = J.n2[x];
                if (y >= 0) { x = y; len += 2; continue; }
            }
            const int y = J.n1[x];
            if (y < 0) break;
            x = y;
            len++;
        }
        if (len < N_SEED) continue;
        W.clen[c] = len;
        chain_ends(W)[c] = x;
    }
}

__global__ void __launch_bounds__(256) k_chain_count(Work W) {
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (blockDim.x >> 5);
    for (int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < W.nbins; b += nw) {
        const int c0 = W.bin_off[b], c1 = W.bin_off[b + 1];
        int cnt = 0;
        for (int c = c0 + lane; c < c1; c += 32 * SWEEP) {
            int len[SWEEP];
#pragma unroll
            for (int j = 0; j < SWEEP; j++) len[j] = c1 - c > 32 * j ? W.clen[c + 32 * j] : 0;
#pragma unroll
            for (int j = 0; j < SWEEP; j++) cnt += len[j] > 0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if (lane == 0) W.bin_cnt[b] = cnt;
    }
}

__global__ void __launch_bounds__(256) k_chain_write(Work W) {
    const int lane = threadIdx.x & 31;
    const int nw = gridDim.x * (blockDim.x >> 5);
    for (int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); b < W.nbins; b += nw) {
        const int c0 = W.bin_off[b], c1 = W.bin_off[b + 1];
        int pos = W.chain_off[b];
        if (lane == 0) {      // the merge counts into these next
            W.bin_cnt[b] = 0;
            if (b % W.nr == 0) W.sec_ymax[b / W.nr] = 0;
        }
        if (W.chain_off[b + 1] == pos) continue;
        for (int base = c0; base < c1; base += 32 * SWEEP) {
            int ln[SWEEP];
#pragma unroll
            for (int j = 0; j < SWEEP; j++) {
                const int c = base + 32 * j + lane;
                ln[j] = c < c1 ? W.clen[c] : 0;
            }
#pragma unroll
            for (int j = 0; j < SWEEP; j++) {
                const int c = base + 32 * j + lane, len = ln[j];
                const unsigned m = __ballot_sync(0xffffffffu, len > 0);
                if (len > 0) {
                    const int p = pos + __popc(m & ((1u << lane) - 1u));
                    if (p < W.cap_chains) {
                        W.chain_start[p] = c;
                        W.chain_last[p] = chain_ends(W)[c];
                        W.chain_len[p] = len;
                        W.chain_bin[p] = b;
                        W.cand_n[p] = len;      // the following adds what it finds and the row range
                        W.cand_rows[p] = 0;
                    } else {
                        set_status(W, ST_CAPACITY);
                    }
                }
                pos += __popc(m);
            }
        }
    }
}

}  // namespace

void launch_chains(const Work &W, cudaStream_t s) {
    const int block = W.tune.block[2] > 0 ? W.tune.block[2] : 256;
    const int warps = block / 32;
    int grid = (W.nbins + warps - 1) / warps;
    if (W.tune.grid[2] > 0 && grid > W.tune.grid[2]) grid = W.tune.grid[2];
    if (grid < 1) grid = 1;
    const int gj = W.sm_count * 8;
    k_mutual<<<gj, 256, 0, s>>>(W);
    int32_t *n1 = reinterpret_cast<int32_t *>(W.claim), *n2 = n1 + (W.n_clusters + 1);
    k_jump<<<gj, 256, 0, s>>>(W, n1, n2);
    k_jump<<<gj, 256, 0, s>>>(W, n2, W.jump4);
    k_chain_walk<<<W.sm_count * 16, 128, 0, s>>>(W);
    k_chain_count<<<grid, block, 0, s>>>(W);
    scan_exclusive(W.bin_cnt, W.chain_off, W.nbins, nullptr, W.counters + CNT_NCHAINS, W.scan_tmp,
                   W.scan_tmp_len, s);
    k_chain_write<<<grid, block, 0, s>>>(W);
}

}  // namespace tpc
