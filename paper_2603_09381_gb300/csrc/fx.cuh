// 60-bit fixed-point complex arithmetic on the integer multipliers, used in
// place of FP64 where a column's norm bounds every entry (Householder QR): the
// FP64 pipe of GB300 does 2 fused multiply-adds per clock and SM.
#pragma once
#include "pm_common.cuh"

// A number x is split as x = h 2^30 + l, -2^29 <= l < 2^29; a product keeps
// h h' + (h l' + l h') / 2^30, rounded, and leaves out l l' / 2^60 (below a
// quarter of a unit, of either sign: with one-sided parts the columns that
// have decayed to a few units would gather a common bias).
struct Fx { int h, l; };
__device__ __forceinline__ Fx fx(long long v) {
  return Fx{(int)((v + (1ll << 29)) >> 30), (int)((unsigned)v << 2) >> 2};
}
__device__ __forceinline__ void fx_mac(long long& hh, long long& cr, Fx a, Fx b) {
  hh += (long long)a.h * b.h;
  cr += (long long)a.h * b.l;
  cr += (long long)a.l * b.h;
}
constexpr long long FX_HALF = 1ll << 29;   // rounds the cross terms' >> 30
__device__ __forceinline__ long long fx_mul(Fx a, Fx b) {
  long long hh = 0, cr = FX_HALF;
  fx_mac(hh, cr, a, b);
  return hh + (cr >> 30);
}
// a + g v, g given as (re, im, -im)
__device__ __forceinline__ longlong2 fx_cfma(longlong2 a, Fx gr, Fx gi, Fx ngi, Fx vr, Fx vi) {
  long long cr = FX_HALF, ci = FX_HALF;
  fx_mac(a.x, cr, gr, vr);
  fx_mac(a.x, cr, ngi, vi);
  fx_mac(a.y, ci, gr, vi);
  fx_mac(a.y, ci, gi, vr);
  a.x += cr >> 30;
  a.y += ci >> 30;
  return a;
}
constexpr double FX_ONE = 1152921504606846976.0;   // 2^60
// x 2^60 / 2^e2 rounded, for |x| < 2^(e2 - 2); subnormal x counts as zero
__device__ __forceinline__ long long fx_from(double x, int e2) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7FF, d = e2 + 1020 - ex;   // d >= 0
  long long m = 0;
  if (ex != 0 && d < 59) {
    m = (long long)(((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 5);
    if (d > 0) m = (m + (1ll << (d - 1))) >> d;
  }
  return (long long)b < 0 ? -m : m;
}
// the double nearest to a 2^(e2 - 60) (|e2| below 900)
__device__ __forceinline__ double fx_to(long long a, int e2) {
  const unsigned long long sign = (unsigned long long)a & 0x8000000000000000ull;
  unsigned long long m = sign ? 0 - (unsigned long long)a : (unsigned long long)a;
  const int lz = __clzll((long long)m);
  m = ((m << (lz & 63)) + 1024) >> 11;   // 53 bits (a carry goes on into the exponent)
  const unsigned long long r = ((unsigned long long)(unsigned)(1023 + 63 - lz - 60 + e2 - 1) << 52) + m;
  return __longlong_as_double((long long)(a == 0 ? 0 : sign | r));
}

// Householder reflector of a column x with first entry alpha and |x|^2 = norm2
// (LAPACK zlarfg's phase: beta real with the sign opposite to Re alpha):
// beta, tau = (beta - alpha) / beta and sc = 1 / (alpha - beta), from one
// reciprocal square root and one reciprocal (the FP64 chain of two square
// roots and four divisions was a quarter of a panel step).  Zeros for x = 0.
__device__ __forceinline__ void fx_reflector(double2 alpha, double norm2, double& beta, double2& tau, double2& sc) {
  beta = 0;
  tau = sc = make_double2(0.0, 0.0);
  if (!(norm2 > 0)) return;
  const double rs = rsqrt(norm2), sg = copysign(1.0, alpha.x);
  double xn = norm2 * rs;
  xn = fma(fma(-xn, xn, norm2), 0.5 * rs, xn);
  beta = -sg * xn;
  tau = make_double2(fma(fabs(alpha.x), rs, 1.0), sg * alpha.y * rs);
  const double dx = alpha.x - beta, inv = 1.0 / fma(dx, dx, alpha.y * alpha.y);
  sc = make_double2(dx * inv, -alpha.y * inv);
}
// Left shift that brings integers of scale 2^e and (true) norm^2 norm2 to a norm in [1/2, 1).
__device__ __forceinline__ int fx_shift(double norm2, int e) {
  const int e2 = (int)((__double2hiint(norm2) >> 20) & 0x7FF) - 1022 - 2 * e;   // in units of the scale: [2^(e2 - 1), 2^e2)
  return norm2 > 0 ? min(max(-((e2 + 1) >> 1), 0), 60) : 0;
}
