// Bessel functions J0, J1, Y0, Y1 of a positive real argument to FP64 accuracy,
// for the Hankel functions H_nu = J_nu + i Y_nu of the Helmholtz kernels.
//
// z >= 8: Hankel's modulus-phase form (DLMF 10.17.3-10.17.4; Abramowitz &
//   Stegun 9.2.5-9.2.10)
//     H_nu(z) = sqrt(2/(pi z)) e^{i w} (P_nu(z) + i Q_nu(z)),  w = z - nu pi/2 - pi/4.
//   What bounds it is the FP64 pipe (2 fused multiply-adds per clock and SM), so
//   P_nu, Q_nu, the reduction of z by pi/2, sine, cosine and their products are
//   computed in 60-bit fixed point on the integer multipliers: every value is
//   below 1.01 and within about 1e-17, a tenth of what the FP64 forms give.
//   FP64 does 1/sqrt(z) from an FP32 estimate (5 operations) and the scaling:
//   12 FP64 operations for one order of about 70 before.  Conversions take an
//   FP64 operation's time each, so they go through the bit patterns as well.
//   - P_nu and z Q_nu: polynomials in 1/z^2 on [8, 12), [12, 20), [20, 30),
//     [30, 60), [60, inf) (hankel_fit.h, written by gen_hankel_fit.py from
//     40-digit values).
//   - sine and cosine of w_0 = z - pi/4 serve both orders (w_1 = w_0 - pi/2).
//   A caller that uses one order pays for one: what it leaves unused is
//   compiled away.
// z < 8: CUDA's j0 / y0 / j1 / y1.
// Complex z (lossy interiors, self blocks): Miller's backward recurrence
//   J_{n-1} = (2n/z) J_n - J_{n+1} from an even start M > |z| + 25 + 3 sqrt|z|,
//   normalised by 1 = J0 + 2 sum J_2k (A&S 9.1.27, 9.1.46), and Neumann's
//   series (A&S 9.1.88)
//     (pi/2) Y0 = (ln(z/2) + gamma) J0 - 2 sum_{k>=1} (-1)^k J_2k / k,
//   with its derivative for Y1 = -Y0':
//     (pi/2) Y1 = -J0/z + (ln(z/2) + gamma) J1 + sum_{k>=1} (-1)^k (J_{2k-1} - J_{2k+1})/k.
#pragma once
#include <cuda_runtime.h>
#include "fx.cuh"
#include "hankel_fit.h"

// below 8: the modulus-phase form does not reach (z >= 0; comparisons of the
// high words, an FP64 one takes a multiplication's time)
__device__ __forceinline__ bool hk_near(double z) { return __double2hiint(z) < 0x40200000; }

// r = sqrt(r2) and ir = 1/r: one FP64 iteration on the estimate gives ir, and
// a last one on r itself its rounding (z = k r is a phase, so that its error
// counts as z times r's); FP32's range is left to sqrt and the division.
__device__ __forceinline__ void hk_distance(double r2, double& r, double& ir) {
  if (!fx_f32_range(r2)) {
    r = sqrt(r2);
    ir = 1.0 / r;
    return;
  }
  ir = fx_rsqrt(r2);
  r = r2 * ir;
  r = fma(fma(-r, r, r2), 0.5 * ir, r);
}

// sin and cos of z - pi/4 in 60-bit fixed point for z >= 8.  With f = z 2/pi =
// n + 1/2 + g/2, |g| <= 1: z - pi/4 = n pi/2 + g pi/4.  z is an integer of 2^-50,
// 2/pi has 96 bits, and f mod 4 is kept to 62 bits: five 32-bit products in
// place of Cody and Waite's FP64 steps.  From z = 8192 up (to about 1e9) whole
// turns are taken off in FP64 first.
__device__ __forceinline__ void hk_sincos_shifted(double z, long long& sn, long long& cs) {
  if (__double2hiint(z) >= 0x40C00000) {
    const double n = rint(z * 0.15915494309189533577) - 4.0;   // leaves z in about [22, 29]
    z = fma(-n, 2.4492935982947064e-16, fma(-n, 6.2831853071795864769, z));
  }
  const unsigned long long b = (unsigned long long)__double_as_longlong(z);
  const int e = (int)(b >> 52) - 1023;                             // 2 .. 12
  const unsigned long long Z = ((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << (e - 2);
  const unsigned z0 = (unsigned)Z, z1 = (unsigned)(Z >> 32);
  const unsigned k2 = 0xA2F9836Eu, k1 = 0x4E441529u, k0 = 0xFC2757D1u;   // 2/pi 2^96
  const unsigned long long lo = (unsigned long long)__umulhi(z0, k1) + __umulhi(z1, k0);
  const unsigned long long m0 = (unsigned long long)z0 * k2 + lo, m = m0 + (unsigned long long)z1 * k1;
  const unsigned long long hi = (unsigned long long)z1 * k2 + (m >> 32) + ((unsigned long long)(m < m0) << 32);
  const unsigned long long f = (hi << 12) | ((unsigned)m >> 20);          // 2^62 to a quadrant, mod 4
  const int n = (int)(f >> 62);
  const long long g = (long long)(f & 0x3FFFFFFFFFFFFFFFull) - (1ll << 61);
  const Fx gf = fx(g >> 1);
  const long long x = fx_mul(gf, gf);
  const int x31 = (int)min(x >> 29, 0x7FFFFFFFll);
  long long s, c;
  hankel_sincos_fit(fx(x), x31, s, c);
  s = fx_mul(fx(s), gf);
  const long long u = (n & 1) ? c : s, v = (n & 1) ? s : c;
  sn = (n & 2) ? -u : u;
  cs = ((n + 1) & 2) ? -v : v;
}

// z >= 8, with iz = 1/z and q = 1/sqrt(z)
__device__ __forceinline__ void hankel_asym(double z, double iz, double q, double& J0, double& Y0, double& J1,
                                            double& Y1) {
  const int zh = __double2hiint(z);
  const double v = iz * iz;
  const long long three = 0x4008000000000000ll;   // 3.0: 3 + x lies in [2, 4)
  long long P0, Q0, P1, Q1;
  auto mapped = [&](double ivh, double sh, int& x31) {
    const long long X = __double_as_longlong(fma(v, ivh, sh)) - three;   // x 2^51
    x31 = (int)(X >> 20);
    return fx(X << 9);
  };
  int x31;
  if (zh >= 0x404E0000) {   // z >= 60
    const Fx x = mapped(HK_IVH4, HK_SH4, x31);
    hankel_fit4(x, x31, P0, Q0, P1, Q1);
  } else if (zh >= 0x403E0000) {   // z >= 30
    const Fx x = mapped(HK_IVH3, HK_SH3, x31);
    hankel_fit3(x, x31, P0, Q0, P1, Q1);
  } else if (zh >= 0x40340000) {   // z >= 20
    const Fx x = mapped(HK_IVH2, HK_SH2, x31);
    hankel_fit2(x, x31, P0, Q0, P1, Q1);
  } else if (zh >= 0x40280000) {   // z >= 12
    const Fx x = mapped(HK_IVH1, HK_SH1, x31);
    hankel_fit1(x, x31, P0, Q0, P1, Q1);
  } else {
    const Fx x = mapped(HK_IVH0, HK_SH0, x31);
    hankel_fit0(x, x31, P0, Q0, P1, Q1);
  }
  // 1/z in 2^-60 (0.375 + 1/z lies in [0.375, 0.5], whose last place is 2^-54)
  const Fx izf = fx((__double_as_longlong(0.375 + iz) - 0x3FD8000000000000ll) << 6);
  long long sn, cs;
  hk_sincos_shifted(z, sn, cs);
  const Fx s = fx(sn), c = fx(cs), ns = fx(-sn), nc = fx(-cs);
  const Fx p0 = fx(P0), q0 = fx(fx_mul(fx(Q0), izf)), p1 = fx(P1), q1 = fx(fx_mul(fx(Q1), izf));
  const double amp = 0.79788456080286535588 * q;     // sqrt(2/pi) / sqrt(z)
  auto two = [&](Fx a0, Fx b0, Fx a1, Fx b1) {
    long long hh = 0, cr = FX_HALF;
    fx_mac(hh, cr, a0, b0);
    fx_mac(hh, cr, a1, b1);
    return amp * fx_to(hh + (cr >> 30), 0);
  };
  J0 = two(p0, c, q0, ns);
  Y0 = two(p0, s, q0, c);
  J1 = two(p1, s, q1, c);
  Y1 = two(q1, s, p1, nc);
}

// The pair of orders at z (below 8 CUDA's j0/y0/j1/y1: ~1e-15 absolute,
// measured against scipy on GB300).
__device__ __forceinline__ void hankel01(double z, double& J0, double& Y0, double& J1, double& Y1) {
  if (!hk_near(z)) {
    const double q = fx_rsqrt(z);
    hankel_asym(z, q * q, q, J0, Y0, J1, Y1);
  } else { J0 = j0(z); Y0 = y0(z); J1 = j1(z); Y1 = y1(z); }
}

// ---- complex argument (lossy interior wavenumbers, self blocks only) ---------------
// Miller / Neumann in complex arithmetic (principal branch of the logarithm);
// valid for moderate |z| and Im z >= 0 (the self blocks need |z| <= k- diam(Gamma)).
__device__ __forceinline__ double2 zmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 zdiv(double2 a, double2 b) {
  const double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 zlog(double2 a) { return make_double2(log(hypot(a.x, a.y)), atan2(a.y, a.x)); }

__device__ __forceinline__ void bessel_complex(double2 z, double2& J0, double2& Y0, double2& J1, double2& Y1) {
  const double az = hypot(z.x, z.y);
  int M = (int)(az + 25.0 + 3.0 * sqrt(az));
  M += (M & 1);
  const double2 t2z = zdiv(make_double2(2.0, 0.0), z);
  double2 jp1 = make_double2(0, 0), jn = make_double2(1e-30, 0);
  double2 norm = make_double2(0, 0), s0 = make_double2(0, 0), s1 = make_double2(0, 0);
  for (int n = M; n >= 1; --n) {
    if ((n & 1) == 0) {
      const int k = n >> 1;
      norm.x += 2.0 * jn.x; norm.y += 2.0 * jn.y;
      const double c = ((k & 1) ? -1.0 : 1.0) / k;
      s0.x += c * jn.x; s0.y += c * jn.y;
    } else {
      const int m = (n + 1) >> 1;
      const double c = (m == 1) ? -1.0 : ((m & 1) ? -1.0 : 1.0) * (1.0 / m + 1.0 / (m - 1));
      s1.x += c * jn.x; s1.y += c * jn.y;
    }
    const double2 a = zmul(make_double2(n * t2z.x, n * t2z.y), jn);
    const double2 jm1 = make_double2(a.x - jp1.x, a.y - jp1.y);
    jp1 = jn;
    jn = jm1;
  }
  norm.x += jn.x; norm.y += jn.y;
  const double2 inv = zdiv(make_double2(1, 0), norm);
  J0 = zmul(jn, inv);
  J1 = zmul(jp1, inv);
  s0 = zmul(s0, inv);
  s1 = zmul(s1, inv);
  double2 lg = zlog(make_double2(0.5 * z.x, 0.5 * z.y));
  lg.x += 0.57721566490153286061;
  const double tp = 0.63661977236758134308;
  const double2 a0 = zmul(lg, J0);
  Y0 = make_double2(tp * (a0.x - 2.0 * s0.x), tp * (a0.y - 2.0 * s0.y));
  const double2 q = zdiv(J0, z), a1 = zmul(lg, J1);
  Y1 = make_double2(tp * (-q.x + a1.x + s1.x), tp * (-q.y + a1.y + s1.y));
}
