// TPC-ITS matching for the drift calibration (arxiv 1712.09434 sections 2.1 and 6: the TPC drift is
// calibrated against tracks of the inner tracker).  Every fitted TPC track (FP32 state and covariance
// at its first hit, in that hit's sector frame) is carried by the exact helix step to x = 0, the
// production vertex, in FP64; an ITS track (global azimuth phi0, z0, tan lambda, q/pT at the vertex
// and their errors) is expressed in the same frame (y = 0, sin phi = sin(phi0 - alpha_k)).  The
// drift calibration is what the match is for, so z only has to fall in a loose window; the match
// chi2 is over (y, sin phi, tan lambda, q/pT) with the TPC covariance plus the ITS errors.  Each side
// keeps its best partner by (floor(chi2 * 2^20), index) (64-bit atomicMin); mutual best pairs are
// matched, and a matched track that starts within the first 8 pad rows, has at least
// 30 hits and |sin phi| < 0.9 at the vertex gets the ITS track's values as its references at the
// vertex (the anchor input of tpc_refit_grad).
//
// What bounds it: FP64, of which this chip has little, and a warp pays for a test however few of its
// lanes are in it.  So the work is split by kind: a
// thread per track for the FP64 step to the vertex; eight lanes a track that pass over the ITS
// tracks of its window in FP32, with margins, and list the pairs that are left (a few per track); a
// thread per listed pair for the FP64 test, so that all lanes of a warp have one.  In one kernel,
// with a thread per track for all of it, almost every candidate of a warp had some lane in the FP64
// test: 766 us on a central event (25,762 x 19,400 tracks); now 22 + 58 + 22 us.
#include "kf.cuh"
#include "tpc_common.cuh"

namespace tpc {

namespace {

constexpr int ITS_NPHI = 360;            // azimuth bins of the ITS track grid
constexpr int ITS_NTL = 12;              // tan lambda bins of 0.2 over [-1.2, 1.2) (outside: the end bins)
constexpr int ITS_NBINS = ITS_NPHI * ITS_NTL;
constexpr double ITS_SIGMA_Y = 0.01;     // y of an ITS track at the vertex (cm)
constexpr double ITS_DPHI = 0.1;         // candidate window in azimuth (rad)
constexpr double ITS_DTL = 0.1;          // candidate window in tan lambda
constexpr double ITS_DZ = 2.0;           // candidate window in z at the vertex (cm)
constexpr double ITS_CHI2 = 100.0;       // chi2 gate of a match (loose: see the header)
// references for the calibration only from matched tracks that start at the inner wall, are long
// and stay well inside the local parametrisation at the vertex (the reference reading)
constexpr int REF_MAX_FIRST_ROW = 8;
constexpr int REF_MIN_HITS = 30;
constexpr double REF_MAX_SNP = 0.9;
constexpr double TWO_PI = 6.283185307179586;

// a - 2 pi n with n the nearest integer (IEEE remainder, exact): [-pi, pi]; no loop, so a corrupt
// angle cannot stall the kernel.  |a| <= pi is its own remainder, so that case skips the call.
__device__ __forceinline__ double wrap_pi(double a) { return fabs(a) <= 0.5 * TWO_PI ? a : remainder(a, TWO_PI); }

__device__ __forceinline__ int tl_bin(float tl) {
    const int b = (int)floorf((tl + 1.2f) * 5.0f);
    return b < 0 ? 0 : (b >= ITS_NTL ? ITS_NTL - 1 : b);
}

__device__ __forceinline__ int phi_bin(double phi) {
    int b = (int)floor(phi / TWO_PI * ITS_NPHI);
    b %= ITS_NPHI;
    return b < 0 ? b + ITS_NPHI : b;
}

constexpr int ITS_REC = 18;      // doubles per track: y, z, snp, tl, q/pT, 4x4 covariance (10), phi, sin, cos alpha
constexpr int ITS_LANES = 8;     // lanes a track takes its window with

struct ItsArgs {
    const float *its;          // [n_its][8]
    int n_its;
    int32_t *match_trk, *match_its;
    float *anchor;             // [n_tracks][8] or nullptr
    double kB, alpha0, dalpha; // curvature constant, sector k centre angle = alpha0 + (k mod half) dalpha
    int32_t *cnt, *off, *fill, *sec;   // sec: 1 if the track may carry references
    unsigned long long *best_trk, *best_its;
    double *sc;                // [n_its][2] sin, cos of phi0
    float4 *srt;               // [n_its][3] ITS tracks in bin order: phi, z, tl, q/pT | s_phi, s_tl, s_q, index | sin, cos
    double *rec;               // [nt_cap][ITS_REC] tracks at the vertex
    int2 *pairs;               // [cap_pairs] (track, ITS track) left for the FP64 test
    int32_t *n_pairs;
    int cap_pairs;
};

__global__ void k_its_count(Work W, ItsArgs A) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *A.n_pairs = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n_its; i += gridDim.x * blockDim.x) {
        const double phi = A.its[8 * (size_t)i];
        atomicAdd(A.cnt + phi_bin(phi) * ITS_NTL + tl_bin(A.its[8 * (size_t)i + 2]), 1);
        A.sc[2 * (size_t)i] = sin(phi);
        A.sc[2 * (size_t)i + 1] = cos(phi);
        A.best_its[i] = ~0ull;
        A.match_its[i] = -1;
    }
}

__global__ void k_its_fill(Work W, ItsArgs A) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n_its; i += gridDim.x * blockDim.x) {
        const float *r = A.its + 8 * (size_t)i;
        const int b = phi_bin(r[0]) * ITS_NTL + tl_bin(r[2]);
        float4 *d = A.srt + 3 * (size_t)(A.off[b] + atomicAdd(A.fill + b, 1));
        d[0] = make_float4(r[0], r[1], r[2], r[3]);
        d[1] = make_float4(r[4], r[6], r[7], __int_as_float(i));
        d[2] = make_float4((float)A.sc[2 * (size_t)i], (float)A.sc[2 * (size_t)i + 1], 0.f, 0.f);
    }
}

// chi2 = d^T M^-1 d for a symmetric positive definite 4x4 M (Cholesky); -1 if M is not
__device__ double chi2_4(double M[4][4], const double d[4]) {
    double L[4][4];
    for (int i = 0; i < 4; i++) {
        for (int j = 0; j <= i; j++) {
            double v = M[i][j];
            for (int k = 0; k < j; k++) v -= L[i][k] * L[j][k];
            if (i == j) {
                if (!(v > 0.0)) return -1.0;
                L[i][i] = sqrt(v);
            } else {
                L[i][j] = v / L[j][j];
            }
        }
    }
    double y[4], c2 = 0.0;
    for (int i = 0; i < 4; i++) {
        double v = d[i];
        for (int k = 0; k < i; k++) v -= L[i][k] * y[k];
        y[i] = v / L[i][i];
        c2 += y[i] * y[i];
    }
    return c2;
}

// The FP64 test of track t (record r) against ITS track i: offers (key, ITS index) to the track and
// (key, track) to the ITS track.
__device__ void its_pair(const ItsArgs &A, int t, int i) {
    const double *q = A.rec + (size_t)t * ITS_REC;
    const float *r = A.its + 8 * (size_t)i;
    const double phi_t = q[15], sa = q[16], ca = q[17];
    if (fabs(wrap_pi((double)r[0] - phi_t)) > ITS_DPHI) return;
    if (fabs((double)r[2] - q[3]) > ITS_DTL || fabs((double)r[1] - q[1]) > ITS_DZ) return;
    // sin, cos of phi0 - alpha from those of phi0 and alpha (no transcendental per pair)
    const double s0 = A.sc[2 * (size_t)i], c0 = A.sc[2 * (size_t)i + 1];
    const double sdp = s0 * ca - c0 * sa, cdp = c0 * ca + s0 * sa;
    const double d[4] = {q[0], q[2] - sdp, q[3] - (double)r[2], q[4] - (double)r[3]};
    const double cph = cdp * (double)r[4];
    const double ev[4] = {ITS_SIGMA_Y * ITS_SIGMA_Y, cph * cph, (double)r[6] * r[6], (double)r[7] * r[7]};
    double M[4][4];
    for (int a = 0, m = 5; a < 4; a++)
        for (int c = 0; c <= a; c++, m++) M[a][c] = M[c][a] = q[m] + (a == c ? ev[a] : 0.0);
    // d^T M^-1 d >= d_a^2 / M_aa for a positive definite M (Cauchy-Schwarz): one component beyond the
    // gate on its own, with a margin far above the rounding of the factorisation, rejects the pair
    // without it (the same decision)
    bool beyond = false;
    for (int a = 0; a < 4; a++) beyond |= d[a] * d[a] > ITS_CHI2 * M[a][a] * (1.0 + 1e-9);
    if (beyond) return;
    const double c2 = chi2_4(M, d);
    if (c2 < 0.0 || c2 > ITS_CHI2) return;
    const unsigned long long k = (unsigned long long)floor(c2 * 1048576.0) << 32;
    atomicMin(A.best_trk + t, k | (unsigned)i);
    atomicMin(A.best_its + i, k | (unsigned)t);
}

// Thread per TPC track: its state and covariance at the vertex in FP64.
__global__ void k_its_state(Work W, ItsArgs A) {
    const DevGeom &g = *W.geom;
    const int nt = min(*W.n_tracks, W.cap_tracks);
    const int nbe = W.ns * W.nr;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
        A.best_trk[t] = ~0ull;
        A.sec[t] = -1;
        if (W.ndf[t] <= 0) continue;
        // sector of the first hit: bin of its cluster by binary search in the bin offsets
        const int off = W.trk_off[t];
        const int h = off >= 0 && off < W.cap_hits ? W.trk_hits[off] : -1;
        if (h < 0 || h >= W.n_clusters) {
            set_status(W, ST_BOUNDS);
            continue;
        }
        int lo = 0, hi = W.nbins - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (W.bin_off[mid] <= h) lo = mid; else hi = mid - 1;
        }
        const int k = (lo % nbe) / W.nr;
        const int first_row = lo % W.nr, n_hits = W.trk_off[t + 1] - off;
        kf::State<double> s;
        s.x = W.xref[t];
        s.frame = k;
        s.rref = 0;
        s.yref = s.zref = 0.0;
        for (int i = 0; i < 5; i++) s.p[i] = W.par[5 * (size_t)t + i];
        for (int i = 0, m = 0; i < 5; i++)
            for (int j = 0; j <= i; j++, m++) s.P[i][j] = s.P[j][i] = W.cov[15 * (size_t)t + m];
        if (!kf::prop_fwd<double>(s, -s.x, A.kB, (double)SNP_MAX)) continue;
        A.sec[t] = first_row <= REF_MAX_FIRST_ROW && n_hits >= REF_MIN_HITS && fabs(s.p[2]) < REF_MAX_SNP;
        const double alpha = A.alpha0 + (k % g.half) * A.dalpha;
        const int ix[4] = {0, 2, 3, 4};
        double *q = A.rec + (size_t)t * ITS_REC;
        for (int i = 0; i < 5; i++) q[i] = s.p[i];
        for (int a = 0, m = 5; a < 4; a++)
            for (int c = 0; c <= a; c++, m++) q[m] = s.P[ix[a]][ix[c]];
        q[15] = alpha + asin(s.p[2]);
        q[16] = sin(alpha);
        q[17] = cos(alpha);
    }
}

// ITS_LANES lanes per track over the ITS tracks of the (azimuth, tan lambda) bins that reach into the
// window; the pairs that the FP32 pre-checks leave go to the list (tested here if it is full).
__global__ void __launch_bounds__(128) k_its_scan(Work W, ItsArgs A) {
    const int nt = min(*W.n_tracks, W.cap_tracks);
    const int sub = threadIdx.x % ITS_LANES;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) / ITS_LANES; t < nt;
         t += gridDim.x * blockDim.x / ITS_LANES) {
        if (A.sec[t] < 0) continue;
        const double *q = A.rec + (size_t)t * ITS_REC;
        const double phi_t = q[15];
        const float tl32 = (float)q[3], z32 = (float)q[1], phi32 = (float)phi_t, sa32 = (float)q[16], ca32 = (float)q[17];
        const float d0_32 = (float)q[0], sn32 = (float)q[2], q32 = (float)q[4];
        const float m0_32 = (float)(q[5] + ITS_SIGMA_Y * ITS_SIGMA_Y), pss32 = (float)q[7];
        const float ptt32 = (float)q[10], pqq32 = (float)q[14];
        const float g = (float)ITS_CHI2 * 1.001f;
        const float mtl = 1e-3f + 1e-6f * fabsf(tl32), mz = 1e-3f + 1e-6f * fabsf(z32);
        const float m2 = 1e-6f * (1.f + fabsf(tl32)), m3 = 1e-6f * (1.f + fabsf(q32));
        auto beyond = [](float d, float m) { return fmaxf(fabsf(d) - m, 0.f); };     // (NaN: 0, left to FP64)
        if (d0_32 * d0_32 > g * m0_32) continue;
        const int b0 = (int)floor((phi_t - ITS_DPHI) / TWO_PI * ITS_NPHI), b1 = (int)floor((phi_t + ITS_DPHI) / TWO_PI * ITS_NPHI);
        // the tan lambda bins that can hold an ITS track within the window (and its margin)
        const int tb0 = tl_bin(tl32 - (float)ITS_DTL - 2e-3f), tb1 = tl_bin(tl32 + (float)ITS_DTL + 2e-3f) + 1;
        for (int bb = b0; bb <= b1; bb++) {
            const int bp = ((bb % ITS_NPHI) + ITS_NPHI) % ITS_NPHI;
            const int j1 = A.off[bp * ITS_NTL + tb1];
            for (int j = A.off[bp * ITS_NTL + tb0] + sub; j < j1; j += ITS_LANES) {
                // FP32 pre-checks that only reject pairs that the FP64 tests reject too: the margins lie far
                // above FP32 rounding, which is relative to the operands (1e-3 and 1e-6 of the value in
                // tan lambda, z and azimuth; 1e-6 and 1e-6 of the value of a component's distance, which
                // the caller's errors may fall below, and 0.1 % of the one-component chi2 bound)
                const float4 r = A.srt[3 * (size_t)j], e = A.srt[3 * (size_t)j + 1], sc = A.srt[3 * (size_t)j + 2];
                if (fabsf(r.z - tl32) > (float)ITS_DTL + mtl || fabsf(r.y - z32) > (float)ITS_DZ + mz) continue;
                float dph = r.x - phi32;
                dph -= rintf(dph * (float)(1.0 / TWO_PI)) * (float)TWO_PI;
                if (fabsf(dph) > (float)ITS_DPHI + 1e-3f + 1e-6f * fabsf(r.x)) continue;
                // distances taken smaller, the error in sin phi larger than they are by the rounding
                const float sdp = sc.x * ca32 - sc.y * sa32, cph = (fabsf(sc.y * ca32 + sc.x * sa32) + 1e-6f) * e.x;
                const float d1 = beyond(sn32 - sdp, 2e-6f), d2 = beyond(tl32 - r.z, m2), d3 = beyond(q32 - r.w, m3);
                if (d1 * d1 > g * (pss32 + cph * cph) || d2 * d2 > g * (ptt32 + e.y * e.y) ||
                    d3 * d3 > g * (pqq32 + e.z * e.z))
                    continue;
                const int i = __float_as_int(e.w);
                // (a full list is not counted on: the count stays near its capacity)
                const int p = __ldcg(A.n_pairs) < A.cap_pairs ? atomicAdd(A.n_pairs, 1) : A.cap_pairs;
                if (p < A.cap_pairs) A.pairs[p] = make_int2(t, i);
                else its_pair(A, t, i);
            }
        }
    }
}

__global__ void __launch_bounds__(128) k_its_pairs(ItsArgs A) {
    const int n = min(*A.n_pairs, A.cap_pairs);
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x)
        its_pair(A, A.pairs[p].x, A.pairs[p].y);
}

__global__ void k_its_link(Work W, ItsArgs A) {
    const int nt = min(*W.n_tracks, W.cap_tracks);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
        const unsigned long long v = A.best_trk[t];
        int m = -1;
        if (v != ~0ull) {
            const int i = (int)(v & 0xffffffffu);
            if (A.best_its[i] == ((v & 0xffffffff00000000ull) | (unsigned)t)) m = i;
        }
        A.match_trk[t] = m;
        if (m >= 0) A.match_its[m] = t;
        if (A.anchor) {
            float *a = A.anchor + 8 * (size_t)t;
            if (A.sec[t] <= 0) m = -1;       // matched, but not a reference of the calibration
            const float *r = A.its + 8 * (size_t)(m >= 0 ? m : 0);
            a[0] = m >= 0 ? (float)ITS_SIGMA_Y : 0.f;
            a[1] = m >= 0 ? r[1] : 0.f;
            a[2] = m >= 0 ? r[5] : 0.f;
            a[3] = m >= 0 ? r[2] : 0.f;
            a[4] = m >= 0 ? r[6] : 0.f;
            a[5] = m >= 0 ? r[3] : 0.f;
            a[6] = m >= 0 ? r[7] : 0.f;
            a[7] = 0.f;
        }
    }
}

}  // namespace

int its_match_nphi() { return ITS_NBINS; }
int its_constants(double *out) {
    const double v[] = {ITS_SIGMA_Y, ITS_DPHI, ITS_DTL, ITS_DZ, ITS_CHI2};
    for (int i = 0; i < 5; i++) out[i] = v[i];
    return 5;
}

void launch_its_match(const Work &W, const float *its, int n_its, int32_t *match_trk, int32_t *match_its,
                      float *anchor, double kB, double alpha0, double dalpha, float *scratch, size_t scratch_words,
                      cudaStream_t s) {
    ItsArgs A;
    A.its = its;
    A.n_its = n_its;
    A.match_trk = match_trk;
    A.match_its = match_its;
    A.anchor = anchor;
    A.kB = kB;
    A.alpha0 = alpha0;
    A.dalpha = dalpha;
    // workspace of the tracking, free between calls: counts, offsets and fill levels of the azimuth
    // bins, the first-hit sector of every track, the best keys
    A.cnt = W.bin_cnt;
    A.off = W.mrg_off;
    A.fill = W.chain_off;
    A.sec = W.trk_n;
    A.best_trk = W.gap_bestT;
    A.best_its = W.gap_bestS;
    A.sc = reinterpret_cast<double *>(W.gap_state);   // 6 words per chain slot >= 2 doubles per ITS track
    // and the workspace of the refit: track records, the sorted ITS tracks, the pair list in the rest
    A.n_pairs = W.counters + CNT_ITS_PAIRS;
    A.rec = reinterpret_cast<double *>(scratch);
    size_t used = (size_t)W.cap_tracks * ITS_REC * 2;
    used = (used + 63) & ~(size_t)63;
    A.srt = reinterpret_cast<float4 *>(scratch + used);
    used += (size_t)n_its * 12;
    A.pairs = reinterpret_cast<int2 *>(scratch + used);
    const size_t left = used < scratch_words ? (scratch_words - used) / 2 : 0;
    A.cap_pairs = (int)(left < (1u << 30) ? left : (1u << 30));
    const int grid = W.sm_count * 4;
    cudaMemsetAsync(A.cnt, 0, sizeof(int32_t) * (ITS_NBINS + 1), s);
    cudaMemsetAsync(A.fill, 0, sizeof(int32_t) * (ITS_NBINS + 1), s);
    k_its_count<<<grid, 256, 0, s>>>(W, A);
    scan_exclusive(A.cnt, A.off, ITS_NBINS, nullptr, nullptr, W.scan_tmp, W.scan_tmp_len, s);
    k_its_fill<<<grid, 256, 0, s>>>(W, A);
    k_its_state<<<grid, 128, 0, s>>>(W, A);
    k_its_scan<<<W.sm_count * 12, 128, 0, s>>>(W, A);
    k_its_pairs<<<grid, 128, 0, s>>>(A);
    k_its_link<<<grid, 256, 0, s>>>(W, A);
}

}  // namespace tpc
