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

// v / 2^d rounded (d >= 0; zero from 63 up), and a sum of squares / 2^(2 d)
__device__ __forceinline__ long long fx_shr(long long v, int d) {
  return d >= 63 ? 0 : (v + ((1ll << d) >> 1)) >> d;
}
__device__ __forceinline__ unsigned __int128 fx_norm_shr(unsigned __int128 v, int d) { return d >= 64 ? 0 : v >> (2 * d); }

// Between positive doubles and floats of the normal FP32 range on the bit
// patterns (truncating): the conversion instructions take an FP64 operation's time.
__device__ __forceinline__ float fx_d2f(double x) {
  return __int_as_float((int)__funnelshift_l((unsigned)__double2loint(x), (unsigned)__double2hiint(x) - 0x38000000u, 3));
}
__device__ __forceinline__ double fx_f2d(float x) {
  const unsigned b = (unsigned)__float_as_int(x);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
// x in [2^-120, 2^120)
__device__ __forceinline__ bool fx_f32_range(double x) {
  return (unsigned)__double2hiint(x) - ((1023u - 120) << 20) < (240u << 20);
}
// 1/sqrt(x) for a positive normal x: Newton's iteration of third order on an
// FP32 estimate q, q (1 - e)^(-1/2) = q (1 + e/2 + 3 e^2/8 + ..), e = 1 - x q^2
// below 2^-20; q^2 is exact.  1/x likewise.  Beyond FP32's range CUDA's.
__device__ __forceinline__ double fx_rsqrt(double x) {
  if (!fx_f32_range(x)) return rsqrt(x);
  const double q = fx_f2d(rsqrtf(fx_d2f(x))), e = fma(-x, q * q, 1.0);
  return fma(q * e, fma(0.375, e, 0.5), q);
}
__device__ __forceinline__ double fx_rcp(double x) {
  if (!fx_f32_range(x)) return 1.0 / x;
  const double y = fx_f2d(1.0f / fx_d2f(x)), e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// The same split at 32 bits, x = h 2^32 + l, which costs two instructions:
// h h' + (h l' + l h') / 2^32 is x x' / 2^64, so the operands carry the factor
// 2^4 between them that 2^-60 numbers need.
__device__ __forceinline__ Fx fw(long long v) { return Fx{(int)((v + 0x80000000ll) >> 32), (int)v}; }
constexpr long long FW_HALF = 1ll << 31;
// a + g v / 2^64, g given as (re, im, -im)
__device__ __forceinline__ longlong2 fw_cfma(longlong2 a, Fx gr, Fx gi, Fx ngi, Fx vr, Fx vi) {
  long long cr = FW_HALF, ci = FW_HALF;
  fx_mac(a.x, cr, gr, vr);
  fx_mac(a.x, cr, ngi, vi);
  fx_mac(a.y, ci, gr, vi);
  fx_mac(a.y, ci, gi, vr);
  a.x += cr >> 32;
  a.y += ci >> 32;
  return a;
}

// The reflector below in integers, for a column in 2^-60 whose norm^2 is
// N 2^-sN: ev with |x| 2^ev in [1/2, 1), and in 2^-60 tau / 2, sc 2^-ev / 2 and
// beta 2^ev.  One reciprocal square root and one reciprocal, each an FP32
// estimate with one third-order Newton step (as in fx_rsqrt): 20 dependent
// integer products, where FP64 took 3,600 cycles.
__device__ __forceinline__ void fx_reflect(long long ar, long long ai, unsigned __int128 N, int sN, int& ev,
                                           longlong2& tau2, longlong2& sc2, long long& beta) {
  ev = 0;
  beta = 0;
  tau2 = sc2 = make_longlong2(0, 0);
  if (N == 0) return;
  const unsigned long long Nh = (unsigned long long)(N >> 64), Nl = (unsigned long long)N;
  const int b = Nh ? 128 - __clzll((long long)Nh) : 64 - __clzll((long long)Nl);
  ev = (sN - b) >> 1;
  const int sh = 64 + 2 * ev - sN;                                           // b + sh: 63 or 64
  const unsigned long long nn = (unsigned long long)(sh >= 0 ? N << sh : N >> -sh);   // |x|^2 2^(2 ev) in 2^-64
  // rs = nn^(-1/2) in (1, 2]
  const float qf = rsqrtf((float)(unsigned)(nn >> 32) * 2.3283064365386963e-10f);
  const unsigned q = (unsigned)(qf * 1073741824.0f);                         // 2^-30
  const unsigned long long q60 = (unsigned long long)q << 30;
  long long e = (1ll << 60) - (long long)__umul64hi(nn, (unsigned long long)q * q);
  int eh = (int)(e >> 14);
  long long e2 = ((long long)eh * eh) >> 32;
  const unsigned long long rs = q60 + (__mul64hi((long long)q60, e << 20) >> 17) + (((long long)(q >> 15) * ((3 * e2) >> 3)) >> 15);
  const unsigned long long xn = __umul64hi(nn, rs);
  const long long one = 1ll << 60;
  const bool nx = ar < 0, ny = ai < 0;
  const unsigned long long ax = min((unsigned long long)((nx ? -ar : ar) << ev), (unsigned long long)one - 1),
                           ay = min((unsigned long long)((ny ? -ai : ai) << ev), (unsigned long long)one - 1);
  const long long ty = (long long)(__umul64hi(ay << 4, rs) >> 1);
  tau2 = make_longlong2((one + (long long)__umul64hi(ax << 4, rs)) >> 1, nx != ny ? -ty : ty);
  beta = nx ? (long long)xn : -(long long)xn;
  // 1 / |alpha - beta|^2, |alpha - beta| 2^ev in [1/2, 2]
  const unsigned long long D = min(ax + xn, 2ull * one - 1), d = __umul64hi(D << 2, D << 2) + __umul64hi(ay << 2, ay << 2);
  const float yf = 1.0f / ((float)(unsigned)(d >> 32) * 3.7252902984619141e-09f);
  const unsigned y = (unsigned)(yf * 268435456.0f);                           // 2^-28
  e = (1ll << 58) - (long long)__umul64hi(d << 1, (unsigned long long)y << 33);
  eh = (int)(e >> 12);
  e2 = ((long long)eh * eh) >> 32;
  const unsigned long long inv =
      ((unsigned long long)y << 32) + (__mul64hi((long long)((unsigned long long)y << 32), e << 22) >> 16) + (((long long)(y >> 13) * e2) >> 15);
  const long long cx = (long long)__umul64hi(D << 3, inv), cy = (long long)__umul64hi(ay << 3, inv);
  sc2 = make_longlong2(nx ? -cx : cx, ny ? cy : -cy);
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
  const double rs = fx_rsqrt(norm2), sg = copysign(1.0, alpha.x);
  double xn = norm2 * rs;
  xn = fma(fma(-xn, xn, norm2), 0.5 * rs, xn);
  beta = -sg * xn;
  tau = make_double2(fma(fabs(alpha.x), rs, 1.0), sg * alpha.y * rs);
  const double dx = alpha.x - beta, inv = fx_rcp(fma(dx, dx, alpha.y * alpha.y));
  sc = make_double2(dx * inv, -alpha.y * inv);
}
// Left shift that brings integers of scale 2^e and (true) norm^2 norm2 to a norm in [1/2, 1).
__device__ __forceinline__ int fx_shift(double norm2, int e) {
  const int e2 = (int)((__double2hiint(norm2) >> 20) & 0x7FF) - 1022 - 2 * e;   // in units of the scale: [2^(e2 - 1), 2^e2)
  return norm2 > 0 ? min(max(-((e2 + 1) >> 1), 0), 60) : 0;
}
