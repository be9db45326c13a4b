// cos and sin of the multiples of an angle in float64, on the integer pipe where that serves.
#pragma once

#include "zp_tri.h"

namespace zp {

// v 2^-62 as a float64, rounded to nearest, by integer operations.
__device__ __forceinline__ double from_fixed62(int64_t v) {
  const uint64_t a = v < 0 ? (uint64_t)-v : (uint64_t)v;
  if (a == 0) return 0.0;
  const int lz = __clzll((long long)a);
  const uint64_t m = a << lz;  // top bit set
  uint64_t b = ((m >> 11) & 0xfffffffffffffull) | ((uint64_t)(1023 - 62 + 63 - lz) << 52);
  b += (m >> 10) & 1;
  return __longlong_as_double((long long)(b | ((uint64_t)v & (1ull << 63))));
}

// The same as a float32 (24 bits of the larger part).
__device__ __forceinline__ float from_split62(const TriTrig& t) { return fmaf((float)t.lo, 0x1p-62f, (float)t.hi * 0x1p-31f); }

// cos and sin of m theta: of the rounded product, turned by what its rounding leaves out (a part of 2^-53 m theta,
// which next to an axis would be all that is left).
__device__ __forceinline__ void sincos_multiple(int m, double th, double* s, double* c) {
  const double p = (double)m * th, e = fma((double)m, th, -p);
  double s0, c0;
  sincos(p, &s0, &c0);
  *s = fma(e, c0, s0);
  *c = fma(-e, s0, c0);
}

// Calls f(m, cos m theta, sin m theta) for m = 0 .. m_max, in T.  In fixed point, with absolute errors below
// (m + 1) 2^-58 (2^-55 measured at m = 32, 2^-53 at 128; a float64 product m theta alone rounds by up to
// 2^-53 m theta), unless the angle is out of range or so close to a multiple of a quarter turn that
// cos or sin of its multiples need relative accuracy: then by angle addition in float64, restarted from
// sincos at every 16th m.  The line: cos and sin both at least 2^-9 (53 bits in fixed point; a quarter of
// a percent of all angles are closer), for float32 results 2^-36 (26 bits).
template <typename T = double, typename F>
__device__ __forceinline__ void for_each_angle(double th, int m_max, F&& f) {
  constexpr bool kFloat = sizeof(T) == sizeof(float);
  int64_t ci = 0, si = 0;
  bool fixed = fabs(th) < 0x1p52;
  if (fixed) {
    tri_cos_sin(tri_turn((uint64_t)__double_as_longlong(th)), ci, si);
    fixed = tri_off_axes(ci, si, kFloat ? 26 : 53);
  }
  if (fixed) {
    const TriTrig c1 = tri_split(ci), s1 = tri_split(si);
    TriTrig c = tri_split(1ll << 62), s = tri_split(0);
    f(0, T(1), T(0));
    for (int m = 1; m <= m_max; ++m) {
      tri_rotate(c, s, c1, s1);
      if constexpr (kFloat)
        f(m, from_split62(c), from_split62(s));
      else
        f(m, from_fixed62((int64_t)c.hi * (1ll << 31) + c.lo), from_fixed62((int64_t)s.hi * (1ll << 31) + s.lo));
    }
  } else if (kFloat && th == 0.0) {
    for (int m = 0; m <= m_max; ++m) f(m, T(1), T(0));
  } else {
    double s1, c1, c = 1.0, s = 0.0;
    sincos(th, &s1, &c1);
    for (int m = 0; m <= m_max; ++m) {
      if (m % 16 == 0) {
        if (m > 0) sincos_multiple(m, th, &s, &c);
      } else {
        const double cn = fma(c, c1, -s * s1);
        s = fma(s, c1, c * s1);
        c = cn;
      }
      f(m, T(c), T(s));
    }
  }
}

}  // namespace zp
