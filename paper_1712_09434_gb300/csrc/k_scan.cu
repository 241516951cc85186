// Device-wide exclusive scan of int32 counts.  Used to turn per-bin chain counts into chain offsets,
// head flags into track ids and per-track hit counts into hit offsets, all without a host round
// trip (counts stay on the device).  Up to ONE_BLOCK counts are scanned by one block, more by two
// launches: tile sums, then every tile adds up the sums in front of it (at most a few thousand
// words from L2) and scans its own counts.  A tracking call makes four scans, and on a single event
// every launch costs about 4 us of a few hundred: a third launch for the tile sums cost more than
// the words read again (one sector 598 -> 562 us together with four resets that other kernels took
// over).
#include "tpc_common.cuh"

namespace tpc {

namespace {

constexpr int SB = 256;           // threads per scan block
constexpr int SI = 8;             // items per thread
constexpr int TILE = SB * SI;

__device__ __forceinline__ int warp_incl(int v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// exclusive scan of one value per thread across the block; the block total goes to *tot
__device__ int block_excl(int v, int *tot) {
    __shared__ int ws[SB / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int inc = warp_incl(v);
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    if (w == 0) {
        const int x = lane < SB / 32 ? ws[lane] : 0;
        const int xi = warp_incl(x);
        if (lane < SB / 32) ws[lane] = xi - x;
        if (lane == 31) *tot = xi;
    }
    __syncthreads();
    const int r = ws[w] + inc - v;
    __syncthreads();
    return r;
}

__device__ __forceinline__ int resolve_n(int n_cap, const int32_t *n_dev) {
    if (!n_dev) return n_cap;
    int n = *n_dev;
    return n < 0 ? 0 : (n > n_cap ? n_cap : n);
}

__global__ void k_scan_reduce(const int32_t *__restrict__ in, int n_cap, const int32_t *n_dev,
                              int32_t *__restrict__ tile_sum) {
    int n = resolve_n(n_cap, n_dev);
    long long base = (long long)blockIdx.x * TILE;
    int s = 0;
    if (base < n) {
        for (int k = 0; k < SI; k++) {
            long long i = base + (long long)k * SB + threadIdx.x;
            if (i < n) s += in[i];
        }
    }
    __shared__ int tot;
    block_excl(s, &tot);
    if (threadIdx.x == 0) tile_sum[blockIdx.x] = base < n ? tot : 0;
}

__global__ void k_scan_apply(const int32_t *__restrict__ in, int32_t *__restrict__ out, int n_cap,
                             const int32_t *n_dev, const int32_t *__restrict__ tile_sum, int32_t *total_dev) {
    int n = resolve_n(n_cap, n_dev);
    long long base = (long long)blockIdx.x * TILE;
    if (base >= n && !(blockIdx.x == 0 && n == 0)) return;
    __shared__ int tot;
    int before = 0;            // the tiles in front
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += SB) before += tile_sum[i];
    block_excl(before, &tot);
    const int off = tot;
    __syncthreads();
    // each thread owns SI consecutive items
    long long i0 = base + (long long)threadIdx.x * SI;
    int v[SI];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SI; k++) {
        long long i = i0 + k;
        v[k] = i < n ? in[i] : 0;
        s += v[k];
    }
    int e = block_excl(s, &tot) + off;
#pragma unroll
    for (int k = 0; k < SI; k++) {
        long long i = i0 + k;
        if (i < n) out[i] = e;
        e += v[k];
    }
    if (threadIdx.x == 0 && base + TILE >= n) {      // the last tile
        out[n] = off + tot;
        if (total_dev) *total_dev = off + tot;
    }
}

// All counts in one block, OT threads, in rounds of OT * SI.
constexpr int OT = 1024;
constexpr int ONE_BLOCK = 2 * OT * SI;
__global__ void __launch_bounds__(OT) k_scan_one(const int32_t *__restrict__ in, int32_t *__restrict__ out, int n_cap,
                                                 const int32_t *n_dev, int32_t *total_dev) {
    __shared__ int ws[OT / 32];
    const int n = resolve_n(n_cap, n_dev);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int carry = 0;
    for (int base = 0; base < n; base += OT * SI) {
        const int i0 = base + threadIdx.x * SI;
        int v[SI], s = 0;
#pragma unroll
        for (int k = 0; k < SI; k++) {
            v[k] = i0 + k < n ? in[i0 + k] : 0;
            s += v[k];
        }
        const int inc = warp_incl(s);
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        const int x = warp_incl(ws[lane]);       // every warp scans the warp totals (OT / 32 = 32 of them)
        const int front = __shfl_sync(0xffffffffu, x, w) - ws[w], all = __shfl_sync(0xffffffffu, x, 31);
        int e = carry + front + inc - s;
#pragma unroll
        for (int k = 0; k < SI; k++) {
            if (i0 + k < n) out[i0 + k] = e;
            e += v[k];
        }
        carry += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[n] = carry;
        if (total_dev) *total_dev = carry;
    }
}

}  // namespace

int scan_tmp_needed(int n_cap) { return (n_cap + TILE - 1) / TILE + 1; }

void scan_exclusive(const int32_t *in, int32_t *out, int n_cap, const int32_t *n_dev, int32_t *total_dev,
                    int32_t *tmp, int tmp_len, cudaStream_t s) {
    (void)tmp_len;
    if (n_cap <= ONE_BLOCK) {
        k_scan_one<<<1, OT, 0, s>>>(in, out, n_cap, n_dev, total_dev);
        return;
    }
    const int n_tiles = (n_cap + TILE - 1) / TILE;
    k_scan_reduce<<<n_tiles, SB, 0, s>>>(in, n_cap, n_dev, tmp);
    k_scan_apply<<<n_tiles, SB, 0, s>>>(in, out, n_cap, n_dev, tmp, total_dev);
}

}  // namespace tpc
