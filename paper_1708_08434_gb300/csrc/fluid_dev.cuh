// fluid_dev.cuh -- arithmetic of the fluid kernels (octree and quadtree):
// the field's square root, table lookups, the Koren limiter and the flux
// through a face, written for the FP64 pipe of this GPU (2 instructions per
// clock and SM): whatever is exact on the bit patterns runs on the integer
// pipe.
#pragma once

#include <math.h>

#include <vector>

#include "sm_internal.cuh"

namespace sm {

// fixed-point index constants of a table of n entries up to e_max, and its
// packed arrays: fc entries {mu, slope, D, slope}, al {alpha, slope}
inline void table_index_consts(Table &tb, const double *packed, int n, double e_max) {
  tb.fc = reinterpret_cast<const double2 *>(packed);
  tb.al = reinterpret_cast<const double2 *>(packed + 4 * 4096);
  int p = 0;
  const double f = frexp(0.5 * ((n - 1) / e_max), &p);  // (n-1)/(2 e_max) = xm 2^(p - 64)
  tb.xm = (unsigned long long)ldexp(f, 64);
  tb.xs = 1035 - p;
  tb.xtop = (unsigned long long)(n - 1) << 51;
  tb.hscale = 0.5 * ((n - 1) / e_max);
}

// the packed arrays of host tables (6 x 4096 doubles)
inline void table_pack(double *out, int n, const double *mu, const double *diff, const double *alpha) {
  const double *src[3] = {mu, diff, alpha};
  for (int k = 0; k < 3; ++k)
    for (int i = 0; i < n; ++i) {
      double *q = k < 2 ? out + 4 * i + 2 * k : out + 4 * 4096 + 2 * i;
      q[0] = src[k][i];
      q[1] = i + 1 < n ? src[k][i + 1] - src[k][i] : 0.0;
    }
}

// Non-negative doubles (no NaN) order as their bit patterns: clamps and
// minima of such values are integer operations, off the FP64 pipe (2 FP64
// instructions per clock and SM on this GPU).
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double dabs(double x) { return __longlong_as_double(dbits(x) & 0x7fffffffffffffffll); }

// bits of a non-negative number (infinity included), 0 for anything else: as
// integers a maximum of these leaves NaNs and negative values out
__device__ __forceinline__ long long size_bits(double x) {
  const unsigned long long b = (unsigned long long)dbits(x);
  return b <= 0x7ff0000000000000ull ? (long long)b : 0ll;
}

// psi(a/b) b for the Koren limiter psi(x) = max(0, min(1, (2+x)/6, x)),
// without the division: 0 when a b <= 0 (a or b is +-0, or their signs
// differ: tested on the bits, with no product), else
// sign(b) min(|b|, (2|b| + |a|)/6, |a|) with the minimum taken on the bit
// patterns
__device__ __forceinline__ double koren(double a, double b) {
  const long long ba = dbits(a), bb = dbits(b);
  if ((ba ^ bb) < 0 || (ba << 1) == 0 || (bb << 1) == 0) return 0.0;
  const double ab = dabs(b), aa = dabs(a);
  long long m = dbits(ab);
  m = min(m, dbits(fma(2.0, ab, aa) * (1.0 / 6.0)));
  m = min(m, dbits(aa));
  return __longlong_as_double(m | (dbits(b) & (long long)0x8000000000000000ull));
}

// Half the table index of a cell, e (n-1)/(2 e_max).  From 2 on in units of
// 2^-51 (rounded; clamped to n - 1): the significand of e times the scale's,
// shifted by the exponents -- integer operations only.  A face's index is then
// the integer sum of its two cells' values, its integer part the top bits; its
// error, 2^-51, is the rounding of an FP64 index from 4 on (a typical index
// of 500 has an ulp of 2^-44).  Below 2, where FP64 is the finer one, the FP64
// product itself with LOW_HALF set in place of its sign.  The FP64 operations
// of such cells are calls: as predicated instructions they take the FP64 pipe
// for every cell (streamer6 field, time step and stage 569 us; 549 as calls).
constexpr unsigned long long LOW_HALF = 1ull << 63;
static __device__ __noinline__ unsigned long long low_half(double e, double scale) {
  return LOW_HALF | (unsigned long long)dbits(e * scale);
}
struct LowIndex {
  double w;
  int i;
};
// (the split itself on the integer pipe: the significand above and below the
// binary point)
static __device__ __noinline__ LowIndex low_split(double yL, double yR, int top) {
  const double y = yL + yR;  // 0 to 4
  const unsigned long long bits = (unsigned long long)dbits(y);
  const int e = (int)(bits >> 52) - 1023;
  if (e < 0) return {y, 0};
  const unsigned long long m = (bits & 0x000fffffffffffffull) | 1ull << 52, f = m << (12 + e);
  const int i = (int)(m >> (52 - e)), lz = __clzll((long long)f);
  if (i >= top) return {0.0, top};
  return {f ? __longlong_as_double((long long)(((unsigned long long)(1021 - lz) << 52) + (f << lz >> 11))) : 0.0, i};
}
__device__ __forceinline__ unsigned long long half_index(double e, const Table &tb) {
  const unsigned long long bits = (unsigned long long)dbits(e);
  const int ex = (int)(bits >> 52);  // the sign included: negative values give a large count
  if (ex & 0x800) return LOW_HALF;
  const unsigned long long A = (bits << 11) | (ex ? 1ull << 63 : 0ull);
  const unsigned long long hi = __umul64hi(A, tb.xm);
  const int sh = tb.xs - (ex ? ex : 1);
  if (sh <= 0) return tb.xtop;
  const unsigned long long x = sh > 63 ? 0ull : ((hi >> (sh - 1)) + 1ull) >> 1;
  if (x >= tb.xtop) return tb.xtop;
  return x < (2ull << 51) ? low_half(e, tb.hscale) : x;
}

// Integer part of the index xL + xR of a face (of a cell: twice its own half),
// clamped to n - 1, and its fraction as an exact double: the leading one of
// the 51 bits is shifted to the hidden bit's place.
__device__ __forceinline__ int index_split(unsigned long long xL, unsigned long long xR, const Table &tb, double &w) {
  unsigned long long x = xL + xR;
  if ((xL | xR) & LOW_HALF) {
    const double yL = __longlong_as_double((long long)(xL & ~LOW_HALF)), yR = __longlong_as_double((long long)(xR & ~LOW_HALF));
    if (xL & xR & LOW_HALF) {  // both in FP64
      const LowIndex r = low_split(yL, yR, (int)(tb.xtop >> 51));
      w = r.w;
      return r.i;
    }
    // the FP64 half to units of 2^-51 (below 2: the shift is at least 0)
    const unsigned long long bits = (xL & LOW_HALF ? xL : xR) & ~LOW_HALF;
    const int sh = 1024 - (int)(bits >> 52);
    const unsigned long long m = (bits & 0x000fffffffffffffull) | 1ull << 52;
    x = (xL & LOW_HALF ? xR : xL) + (sh > 54 ? 0ull : ((m << 1 >> sh) + 1ull) >> 1);
  }
  x = x < tb.xtop ? x : tb.xtop;
  const unsigned long long f = x & ((1ull << 51) - 1ull);
  const int lz = __clzll((long long)f);  // 13 .. 63 when f != 0
  const unsigned long long m = f << (lz - 11);
  w = f ? __longlong_as_double((long long)(((unsigned long long)(1034 - lz) << 52) + m)) : 0.0;
  return (int)(x >> 51);
}

// dx times the flux through the face between cells L and R (positive
// toward R): v = -mu(E*) E_face with E_face = (p_L - p_R)/dx, E* = (|E|_L +
// |E|_R)/2; advective part by Eq. 7 when v >= 0 and Eq. 6 when v < 0; diffusive
// part -D(E*) (n_R - n_L)/dx.  Written as -mu dp n_f - D dn: v < 0 exactly when
// mu dp > 0; from the differences
// n_L - n_L2, n_R - n_L and n_R2 - n_R, which a line of faces shares, and the
// half table indices of the two cells
__device__ __forceinline__ double face_flux_d(double nL, double nR, double dm, double dn, double dq, double dp,
                                              unsigned long long xL, unsigned long long xR, const Table &tb) {
  double w;
  const double2 *fc = tb.fc + 2 * index_split(xL, xR, tb, w);
  const double2 cm = __ldg(fc), cd = __ldg(fc + 1);
  const double t1 = fma(w, cm.y, cm.x) * dp;
  const bool up = dbits(t1) > 0;  // v < 0: the upwind cell is R
  const double k = koren(up ? dq : dm, dn);
  const double nf = (up ? nR : nL) + __longlong_as_double(dbits(k) ^ (up ? (long long)0x8000000000000000ull : 0ll));
  return fma(-t1, nf, -fma(w, cd.y, cd.x) * dn);
}

// x / 2, exactly, on the integer pipe for zeros and values whose half is a
// normal number
__device__ __forceinline__ double halve(double x) {
  const long long b = dbits(x);
  const int ex = (int)((unsigned long long)b >> 52) & 0x7ff;
  if ((ex > 1 && ex < 0x7ff)) return __longlong_as_double(b - (1ll << 52));
  return (b << 1) == 0 ? x : 0.5 * x;
}

// sqrt(x) with four FP64 instructions: x = 4^k m, 1 <= m < 4, from the bits;
// g = sqrt(m) and h = 1/(2 sqrt(m)) in single precision; two steps of
// Newton's iteration g += (m - g^2) h (Heron's method with the division
// replaced by the approximate reciprocal), which leave an error of 2^-65
// beside the last rounding.  Zeros, subnormals, infinities, NaNs and negative
// values take the library function.
__device__ __forceinline__ double sqrt_newton(double x) {
  const unsigned long long bits = (unsigned long long)dbits(x);
  const int ex = (int)(bits >> 52);
  if (ex == 0 || ex >= 0x7ff) return (bits << 1) == 0 ? x : sqrt(x);
  const int odd = (ex - 1023) & 1, k = (ex - 1023 - odd) / 2;
  const double m = __longlong_as_double((long long)((bits & 0x000fffffffffffffull) | (unsigned long long)(1023 + odd) << 52));
  const float mf = __uint_as_float((unsigned)(127 + odd) << 23 | (unsigned)((bits >> 29) & 0x7fffffu));
  const float rs = rsqrtf(mf);
  const double g0 = cvt_f32_f64(mf * rs), h = cvt_f32_f64(0.5f * rs);
  const double g1 = fma(fma(-g0, g0, m), h, g0);
  const double g2 = fma(fma(-g1, g1, m), h, g1);
  return __longlong_as_double(dbits(g2) + ((long long)k << 52));
}

}  // namespace sm
