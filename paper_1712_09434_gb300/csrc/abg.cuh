// Integer steady-state Kalman filter of the following (alpha-beta-gamma = 1/2, 1/8, 1/32 on a Q16
// state, floor shifts; arxiv 1712.09434 section 3: Kalman-filter track following).  Header-only and
// free of CUDA, so that the two widths can be compared on the host.
//
// The filter word T is int64, or int32 for geometries with ymax <= 16383 and zmax <= 32767 (narrow):
// then a Q16 coordinate fits 32 bits, with Z shifted by -16384 so that one step never carries a
// prediction past the word (a step moves less than 16384 LSB: the velocity that a track can build
// up inside the drift range at 343 LSB per residual stays below that).  Sums and differences are
// taken modulo 2^32 (unsigned; a signed overflow would be undefined), so only the reading of a
// prediction could be wrong, for a hit more than 16384 LSB beyond the drift range; such a chain is not
// extended (it would stop at once).
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define ABG_HD __host__ __device__ __forceinline__
#else
#define ABG_HD inline
#endif

namespace tpc {

constexpr int NARROW_YMAX = 16383, NARROW_ZMAX = 32767, NARROW_ZHIT = 49151;

// a + b and a - b, in 32 bits modulo 2^32
ABG_HD int32_t wrap_add(int32_t a, int32_t b) { return (int32_t)((uint32_t)a + (uint32_t)b); }
ABG_HD int32_t wrap_sub(int32_t a, int32_t b) { return (int32_t)((uint32_t)a - (uint32_t)b); }
ABG_HD long long wrap_add(long long a, long long b) { return a + b; }
ABG_HD long long wrap_sub(long long a, long long b) { return a - b; }

template <class T>
struct Abg {
    static constexpr int ZB = sizeof(T) == 4 ? 16384 : 0;   // Z as the filter holds it: z - ZB
    T p, v, a;
};
template <class T>
ABG_HD T q16(int m) {
    if constexpr (sizeof(T) == 4) return (T)((uint32_t)m << 16);
    else return (T)m * 65536;
}

// state at m0 with the velocity of the step to m1, drow = 1 or 2 rows further (2 across a row that
// a link skips; the division is exact)
template <class T>
ABG_HD void abg_init(Abg<T> &f, int m0, int m1, int drow) {
    f.p = q16<T>(m0);
    f.v = (T)(m1 - m0) * (65536 / drow);
    f.a = 0;
}
// position one row further
template <class T>
ABG_HD T abg_ahead(const Abg<T> &f) {
    return wrap_add(f.p, wrap_add(f.v, (T)(f.a >> 1)));
}
template <class T>
ABG_HD void abg_predict(Abg<T> &f) {
    f.p = abg_ahead(f);
    f.v = wrap_add(f.v, f.a);
}
template <class T>
ABG_HD void abg_update(Abg<T> &f, int m) {
    const T e = wrap_sub(q16<T>(m), f.p);
    f.p = wrap_add(f.p, (T)(e >> 1));
    f.v = wrap_add(f.v, (T)(e >> 3));
    f.a = wrap_add(f.a, (T)(e >> 5));
}
template <class T>
ABG_HD int q16_round(T p) {
    return (int)(wrap_add(p, (T)32768) >> 16);
}

}  // namespace tpc
