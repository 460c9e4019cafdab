// Column-pivoted Householder QR, one launch per elimination step.
//
// Each CTA owns up to 16 columns of one matrix.  The step's pivot (largest
// trailing norm; norms within a factor 1 - 1e-12 of the largest count as tied
// and the lowest column index wins) and its Householder reflector (LAPACK
// zlarfg phase convention) are read from the matrix's CpqrPick, written at
// the end of the previous step by the matrix's last CTA to finish: choosing
// them anew in every CTA cost more than the columns (square roots, divisions
// and comparisons on the FP64 pipe, 10 us of an SM per step).  The CTA applies
// H^H to its columns, recomputing their trailing norms from scratch.  The
// pivot column itself is left in place; R_ss goes to rdiag[s].  Because
// consecutive steps are consecutive launches no grid-wide barrier is needed.
//
// complex128 columns are held in 60-bit fixed point (fx.cuh, one power-of-two
// scale per column from its initial norm): a reflection keeps a column's
// norm, and the integer multipliers do a complex multiply-add in a quarter of
// the FP64 pipe's time.  The pivot column enters the dot products shifted up
// to its norm, and the trailing norms are sums of exact 120-bit squares, so
// both keep a double's relative accuracy however far a column has decayed.
#include "cpqr.cuh"
#include "fx.cuh"
#include "prof.cuh"
#include <algorithm>
#include <cooperative_groups.h>
#include <atomic>
#include <mutex>

namespace {

constexpr double TIE = 1e-12;

template <typename C>
__global__ void __launch_bounds__(256) k_init_norms(const CpqrProb<C>* __restrict__ P, const CpqrChunk* __restrict__ chunks) {
  typedef typename real_of<C>::type R;
  const CpqrChunk ch = chunks[blockIdx.x];
  const CpqrProb<C> p = P[ch.id];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int c = ch.c0 + warp; c < ch.c1; c += 8) {
    C* col = p.Z + (size_t)c * p.ld;
    R acc = 0;
    for (int r = lane; r < p.W; r += 32) acc += abs2(col[r]);
    acc = warp_sum(acc);
    if (lane == 0) p.norm2[c] = (double)acc;
    if constexpr (sizeof(C) == 16) {
      // to fixed point, the norm brought into (1/8, 1/4] (a column that is not finite: zeros, and *bad)
      int e = 0;
      const bool ok = isfinite(acc);
      if (ok && acc > 0) frexp(sqrt(acc) * (1.0 + 1e-9), &e);
      e += 2;
      longlong2* f = reinterpret_cast<longlong2*>(col);
      for (int r = lane; r < p.W; r += 32) {
        const double2 z = col[r];
        f[r] = make_longlong2(ok ? fx_from(z.x, e) : 0, ok ? fx_from(z.y, e) : 0);
      }
      if (lane == 0) {
        p.cexp[c] = e;
        if (!ok) *p.bad = 1;
      }
    }
  }
}

__device__ __forceinline__ double ld_norm(const double* p) { return __ldcg(p); }

// Pivot and reflector of step s (the matrix's norms of step s are complete),
// or the end of the phase.  All 256 threads of one CTA.  Norms are compared
// as integers (non-negative doubles order like their bit patterns).
template <typename C>
__device__ void cpqr_pick(const CpqrProb<C>& p, int s) {
  typedef typename real_of<C>::type R;
  typedef unsigned long long u64;
  __shared__ u64 s_k[8];
  __shared__ int s_i[8];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = p.n;
  const double* cur = p.norm2 + (s & 1) * n;
  auto key_of = [&](int c) -> u64 {   // 0: pivoted (negative) or not a number
    const u64 b = (u64)__double_as_longlong(ld_norm(cur + c));
    return b <= 0x7FF0000000000000ull ? b + 1 : 0;
  };
  u64 k = 0;
  if (s < p.target)
    for (int c = tid; c < n; c += 256) { const u64 x = key_of(c); k = x > k ? x : k; }
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
  if (lane == 0) s_k[warp] = ((u64)hi << 32) | lo;
  __syncthreads();
  k = s_k[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) k = s_k[w] > k ? s_k[w] : k;
  const double mx = k ? __longlong_as_double((long long)(k - 1)) : 0.0;
  // lowest index within the tie band
  const u64 band = k ? (u64)__double_as_longlong((1.0 - TIE) * mx) + 1 : ~0ull;
  int qi = n;
  if (k)
    for (int c = tid; c < n; c += 256) if (key_of(c) >= band) { qi = c; break; }
  qi = __reduce_min_sync(0xffffffffu, qi);
  if (lane == 0) s_i[warp] = qi;
  __syncthreads();
  if (warp != 0) return;
  qi = s_i[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) qi = min(qi, s_i[w]);
  CpqrPick<C> pk{};
  pk.q = -1;
  bool go = k != 0 && qi < n;
  if (go && p.mode == CPQR_FIND_RANK) {
    const double ref = s == 0 ? sqrt(mx) : *p.ref;
    if (s == 0 && lane == 0) *p.ref = ref;
    if (!(sqrt(mx) > p.tol * ref)) {
      if (lane == 0) *p.rank = s;
      go = false;
    }
  }
  if (go) {
    pk.q = qi;
    const double nq = ld_norm(cur + qi);
    C tau = czero<C>();
    if constexpr (sizeof(C) == 16) {
      const int eq = p.cexp[qi];
      const longlong2 a = __ldcg(reinterpret_cast<const longlong2*>(p.Z + s + (size_t)qi * p.ld));
      const double2 alpha = make_double2(fx_to(a.x, 0), fx_to(a.y, 0));   // in units of the column's scale
      double beta;
      double2 sc;
      const double nn = ldexp(nq, -2 * eq);
      fx_reflector(alpha, nn, beta, tau, sc);
      pk.ev = fx_shift(nq, eq);   // x 2^ev below 1, sc 2^-ev at most 2
      pk.sc = __longlong_as_double((long long)(1023 - pk.ev) << 52) * sc;
      pk.csc = __longlong_as_double((long long)(1023 - 60 - pk.ev) << 52) * conj(sc);   // applied to the shifted sums
      // A factorization continued past its rank can meet a column whose integers
      // are all zero: R_ss is then the unit of its scale, not zero, so that
      // the interpolation matrix stays finite.
      pk.beta = make_double2(ldexp(beta != 0 ? beta : 0x1p-58, eq), 0.0);
    } else {
      const C alpha = __ldcg(p.Z + s + (size_t)qi * p.ld);
      const R xnorm = (R)sqrt(nq);
      const R beta = -copysign(xnorm, alpha.x);
      C sc = czero<C>();
      pk.reflect = xnorm > 0;
      if (pk.reflect) {
        const C bm = mk(beta, (R)0);
        tau = cdiv(bm - alpha, bm);
        sc = cdiv(mk((R)1, (R)0), alpha - bm);
      }
      pk.sc = sc;
      pk.csc = conj(sc);
      pk.beta = mk(beta, (R)0);
    }
    pk.ctau = conj(tau);
    if (lane == 0) {
      p.rdiag[s] = pk.beta;
      p.perm[s] = qi;
    }
  }
  if (lane == 0) *p.pick = pk;
}

// First pivot of a phase (step `base` of every matrix).
template <typename C>
__global__ void __launch_bounds__(256) k_cpqr_start(const CpqrProb<C>* __restrict__ P) {
  const CpqrProb<C> p = P[blockIdx.x];
  cpqr_pick<C>(p, p.base);
  if (threadIdx.x == 0) *p.done = 0;
}

// Sum of one value over the 256 threads of the CTA (every thread gets it).
template <typename R>
__device__ __forceinline__ R block_sum(R v, R* sh) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  R t = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) t += sh[w];
  return t;
}

// The chunk's columns one at a time, each held by the whole CTA in registers
// (RPT rows per thread): one read and one write of every trailing entry, with
// all of a thread's loads in flight together.  Requires W - s - 1 <= 256 RPT.
template <typename C, int RPT>
__device__ void cta_columns(const CpqrProb<C>& p, const CpqrChunk& ch, int s, int q, const C* xq, C ctau, C csc,
                            C sc, const double* cur, double* nxt) {
  typedef typename real_of<C>::type R;
  __shared__ R shx[8], shy[8], shn[8];
  const int tid = threadIdx.x;
  for (int c = ch.c0; c < ch.c1; ++c) {
    if (cur[c] < 0 || c == q) { if (tid == 0) nxt[c] = -1.0; continue; }
    C* col = p.Z + (size_t)c * p.ld;
    C v[RPT];
    C dot = czero<C>();
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = s + 1 + tid + 256 * i;
      v[i] = (r < p.W) ? col[r] : czero<C>();
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = s + 1 + tid + 256 * i;
      if (r < p.W) cfma_conj(dot, __ldg(&xq[r]), v[i]);
    }
    dot.x = block_sum(dot.x, shx);
    dot.y = block_sum(dot.y, shy);
    const C a_s = col[s];
    const C d = a_s + csc * dot;     // v^H a with v = [1; x/(alpha - beta)]
    const C f = ctau * d;            // H^H a = a - conj(tau) v (v^H a)
    const C fs = f * sc;
    R e = 0;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = s + 1 + tid + 256 * i;
      if (r < p.W) {
        cfms(v[i], fs, __ldg(&xq[r]));
        col[r] = v[i];
        e += abs2(v[i]);
      }
    }
    e = block_sum(e, shn);
    if (tid == 0) {
      col[s] = a_s - f;
      nxt[c] = (double)e;
    }
    __syncthreads();
  }
}

// One elimination step of a complex64 chunk's columns (all 256 threads of
// the CTA take the same path through the barriers).
template <typename C, bool TALL>
__device__ void cpqr_columns(const CpqrProb<C>& p, const CpqrChunk& ch, int s, const CpqrPick<C>& pk) {
  typedef typename real_of<C>::type R;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = p.n, q = pk.q;
  const double* cur = p.norm2 + (s & 1) * n;
  double* nxt = p.norm2 + ((s + 1) & 1) * n;
  const C* xq = p.Z + (size_t)q * p.ld;
  const C ctau = pk.ctau, sc = pk.sc, csc = pk.csc;
  const bool reflect = pk.reflect;
  // complex64 tall enough to fill the CTA (short columns are barrier-bound) and fitting in registers
  if (TALL && sizeof(C) == 8 && reflect && p.W >= 2048 && p.W <= 256 * 32) {
    cta_columns<C, 32>(p, ch, s, q, xq, ctau, csc, sc, cur, nxt);
    return;
  }
  for (int c = ch.c0 + warp; c < ch.c1; c += 8) {
    if (cur[c] < 0 || c == q) { if (lane == 0) nxt[c] = -1.0; continue; }
    C* col = p.Z + (size_t)c * p.ld;
    if (!reflect) {
      R acc = 0;
      for (int r = s + 1 + lane; r < p.W; r += 32) acc += abs2(col[r]);
      acc = warp_sum(acc);
      if (lane == 0) nxt[c] = (double)acc;
      continue;
    }
    // four independent partial sums keep several loads in flight per lane
    C d0 = czero<C>(), d1 = czero<C>(), d2 = czero<C>(), d3 = czero<C>();
    int r = s + 1 + lane;
    for (; r + 96 < p.W; r += 128) {
      const C x0 = __ldg(&xq[r]), x1 = __ldg(&xq[r + 32]), x2 = __ldg(&xq[r + 64]), x3 = __ldg(&xq[r + 96]);
      const C a0 = col[r], a1 = col[r + 32], a2 = col[r + 64], a3 = col[r + 96];
      cfma_conj(d0, x0, a0); cfma_conj(d1, x1, a1); cfma_conj(d2, x2, a2); cfma_conj(d3, x3, a3);
    }
    for (; r < p.W; r += 32) cfma_conj(d0, __ldg(&xq[r]), col[r]);
    C dot = (d0 + d1) + (d2 + d3);
    dot.x = warp_sum(dot.x); dot.y = warp_sum(dot.y);
    const C a_s = col[s];
    __syncwarp();                   // every lane has read col[s] before lane 0 rewrites it
    dot = a_s + csc * dot;          // v^H a with v = [1; x/(alpha - beta)]
    const C f = ctau * dot;         // H^H a = a - conj(tau) v (v^H a)
    const C fs = f * sc;
    if (lane == 0) col[s] = a_s - f;
    R e0 = 0, e1 = 0, e2 = 0, e3 = 0;
    r = s + 1 + lane;
    for (; r + 96 < p.W; r += 128) {
      C v0 = col[r], v1 = col[r + 32], v2 = col[r + 64], v3 = col[r + 96];
      cfms(v0, fs, __ldg(&xq[r])); cfms(v1, fs, __ldg(&xq[r + 32]));
      cfms(v2, fs, __ldg(&xq[r + 64])); cfms(v3, fs, __ldg(&xq[r + 96]));
      col[r] = v0; col[r + 32] = v1; col[r + 64] = v2; col[r + 96] = v3;
      e0 += abs2(v0); e1 += abs2(v1); e2 += abs2(v2); e3 += abs2(v3);
    }
    for (; r < p.W; r += 32) {
      C v = col[r];
      cfms(v, fs, __ldg(&xq[r]));
      col[r] = v;
      e0 += abs2(v);
    }
    R acc = (e0 + e1) + (e2 + e3);
    acc = warp_sum(acc);
    if (lane == 0) nxt[c] = (double)acc;
  }
}

// Sums over the warp of a 59-bit signed integer, 24 bits at a time, as two
// words whose value is hi 2^24 + lo.
__device__ __forceinline__ void warp_sum_parts(long long x, long long& hi, unsigned& lo) {
  lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0xFFFFFFu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 24) & 0xFFFFFFu);
  const int top = __reduce_add_sync(0xffffffffu, (int)(x >> 48));
  hi = ((long long)top << 24) + mid;
}

// d += conj(x) (a 2^ea).  Both are shifted up to their norms, so that the sum
// has a double's accuracy relative to them: a factorization continued far past
// its rank works on columns of a few units, and row entries that are off by as
// much as the pivot make the interpolation matrix grow with every step.
__device__ __forceinline__ void fx_dot(longlong2& d, longlong2 x, longlong2 a, int ea) {
  const Fx xr = fx(x.x), xi = fx(x.y), nxi = fx(-x.y), ar = fx(a.x << ea), ai = fx(a.y << ea);
  long long cr = FX_HALF, ci = FX_HALF;
  fx_mac(d.x, cr, xr, ar); fx_mac(d.x, cr, xi, ai);
  fx_mac(d.y, ci, xr, ai); fx_mac(d.y, ci, nxi, ar);
  d.x += cr >> 30;
  d.y += ci >> 30;
}
// From the sum x^H a (parts of warp_sum_parts) over the rows below s: the entry
// a_s is updated and the factor of the rows below formed, a += g (x 2^ev): |f| is
// at most 1/2 (a reflection moves a by at most twice its norm of 1/4), so |g| at most 1.
__device__ __forceinline__ void fx_factor(double2 ctau, double2 csc, double2 sc, longlong2 h, uint2 l, int ea,
                                          longlong2* a_s, int4& g, int2& gn) {
  const longlong2 as = *a_s;
  const double u = __longlong_as_double((long long)(1023 - ea) << 52);
  const double2 dot = make_double2(u * ((double)h.x * 16777216.0 + (double)l.x), u * ((double)h.y * 16777216.0 + (double)l.y));
  const double2 f = ctau * (make_double2(fx_to(as.x, 0), fx_to(as.y, 0)) + csc * dot);   // conj(tau) v^H a
  *a_s = make_longlong2(as.x - __double2ll_rn(f.x * FX_ONE), as.y - __double2ll_rn(f.y * FX_ONE));
  const double2 t = -(f * sc);
  const long long ti = __double2ll_rn(t.y * FX_ONE);
  const Fx r = fx(__double2ll_rn(t.x * FX_ONE)), i = fx(ti), ni = fx(-ti);
  g = make_int4(r.h, r.l, i.h, i.l);
  gn = make_int2(ni.h, ni.l);
}
__device__ __forceinline__ longlong2 fx_update(longlong2 a, longlong2 x, int4 g, int2 gn) {
  return fx_cfma(a, Fx{g.x, g.y}, Fx{g.z, g.w}, Fx{gn.x, gn.y}, fx(x.x), fx(x.y));
}
// Exact sum of squares of integers below 2^58: a = h 2^29 + l, 0 <= l < 2^29,
// sums of h^2, h l and l^2, folded before they can overflow (every 8 entries).
struct FxSquares {
  long long A = 0, B = 0, D = 0;
  __device__ __forceinline__ void part(long long v) {
    const int h = (int)(v >> 29), l = (int)v & 0x1FFFFFFF;
    A += (long long)h * h;
    B += (long long)h * l;
    D += (long long)l * l;
  }
  __device__ __forceinline__ void add(longlong2 a) { part(a.x); part(a.y); }
  // the sum is A 2^58 + B 2^30 + D
  __device__ __forceinline__ void fold() {
    B += D >> 30; D &= 0x3FFFFFFF;
    A += B >> 28; B &= 0xFFFFFFF;
  }
  // over the warp: x 2^58 + y
  __device__ __forceinline__ longlong2 warp_total() {
    fold();
    longlong2 t;
    long long h;
    unsigned l;
    warp_sum_parts(A, h, l);
    t.x = (h << 24) + l;
    warp_sum_parts((B << 30) + D, h, l);
    t.y = (h << 24) + l;
    return t;
  }
};
// (x 2^58 + y) 2^-120 scale^2
__device__ __forceinline__ double fx_norm2(longlong2 w, int e) {
  return ldexp(fma((double)w.x, 0x1p58, (double)w.y), 2 * e - 120);
}

// One elimination step of a complex128 chunk's columns in fixed point, two
// columns per warp: dot products with the shifted pivot column; the chunk's
// factors at once, a thread per column (a warp's FP64 instruction costs the
// same for one lane as for 32); the update and the exact squares of the new
// entries; the chunk's norms at once.
__device__ void cpqr_columns_fx(const CpqrProb<double2>& p, const CpqrChunk& ch, int s, const CpqrPick<double2>& pk) {
  static_assert(CPQR_CB == 16, "two columns per warp");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = p.n, q = pk.q, W = p.W, ev = pk.ev;
  const double* cur = p.norm2 + (s & 1) * n;
  double* nxt = p.norm2 + ((s + 1) & 1) * n;
  __shared__ longlong2 s_dot[CPQR_CB], s_nrm[CPQR_CB];
  __shared__ uint2 s_dlo[CPQR_CB];
  __shared__ int4 s_g[CPQR_CB];
  __shared__ int2 s_gn[CPQR_CB];
  const longlong2* xq = reinterpret_cast<const longlong2*>(p.Z + (size_t)q * p.ld);
  const int c0 = ch.c0 + warp, c1 = c0 + 8;
  const bool on0 = c0 < ch.c1 && c0 != q && !(cur[c0] < 0), on1 = c1 < ch.c1 && c1 != q && !(cur[c1] < 0);
  longlong2* a0 = reinterpret_cast<longlong2*>(p.Z + (size_t)c0 * p.ld);
  longlong2* a1 = reinterpret_cast<longlong2*>(p.Z + (size_t)c1 * p.ld);
  const longlong2 zero = make_longlong2(0, 0);
  if (on0 || on1) {
    const int e0 = on0 ? fx_shift(cur[c0], p.cexp[c0]) : 0, e1 = on1 ? fx_shift(cur[c1], p.cexp[c1]) : 0;
    longlong2 d0 = zero, d1 = zero;
#pragma unroll 2
    for (int r = s + 1 + lane; r < W; r += 32) {
      const longlong2 x = xq[r], y0 = on0 ? a0[r] : zero, y1 = on1 ? a1[r] : zero;
      const longlong2 xs = make_longlong2(x.x << ev, x.y << ev);
      fx_dot(d0, xs, y0, e0);
      fx_dot(d1, xs, y1, e1);
    }
    longlong2 h;
    uint2 l;
    warp_sum_parts(d0.x, h.x, l.x); warp_sum_parts(d0.y, h.y, l.y);
    if (lane == 0) { s_dot[warp] = h; s_dlo[warp] = l; }
    warp_sum_parts(d1.x, h.x, l.x); warp_sum_parts(d1.y, h.y, l.y);
    if (lane == 0) { s_dot[warp + 8] = h; s_dlo[warp + 8] = l; }
  }
  __syncthreads();
  const int c = ch.c0 + tid;
  const bool mine = tid < CPQR_CB && c < ch.c1 && c != q && !(cur[c] < 0);
  if (mine)
    fx_factor(pk.ctau, pk.csc, pk.sc, s_dot[tid], s_dlo[tid], fx_shift(cur[c], p.cexp[c]),
              reinterpret_cast<longlong2*>(p.Z + s + (size_t)c * p.ld), s_g[tid], s_gn[tid]);
  __syncthreads();
  if (on0 || on1) {
    const int4 g0 = s_g[warp], g1 = s_g[warp + 8];
    const int2 n0 = s_gn[warp], n1 = s_gn[warp + 8];
    FxSquares q0, q1;
    int it = 0;
#pragma unroll 2
    for (int r = s + 1 + lane; r < W; r += 32) {
      const longlong2 x = xq[r], xs = make_longlong2(x.x << ev, x.y << ev);
      if (on0) { const longlong2 v = fx_update(a0[r], xs, g0, n0); a0[r] = v; q0.add(v); }
      if (on1) { const longlong2 v = fx_update(a1[r], xs, g1, n1); a1[r] = v; q1.add(v); }
      if ((++it & 7) == 0) { q0.fold(); q1.fold(); }
    }
    longlong2 w = q0.warp_total();
    if (lane == 0) s_nrm[warp] = w;
    w = q1.warp_total();
    if (lane == 0) s_nrm[warp + 8] = w;
  }
  __syncthreads();
  if (tid < CPQR_CB && c < ch.c1) nxt[c] = mine ? fx_norm2(s_nrm[tid], p.cexp[c]) : -1.0;
}

// Persistent grid (a multiple of the SM count): CTAs take chunks from a
// per-launch counter, largest matrices first, until none is left.  TALL
// compiles in the register-resident path for tall complex64 columns; without
// it the kernel needs far fewer registers (more resident CTAs), which is what
// the n x n triangles of the QR-first path want.  The CTA that finishes a
// matrix's last chunk picks the next step's pivot.
template <typename C, bool TALL>
__global__ void __launch_bounds__(256) k_cpqr_step(const CpqrProb<C>* __restrict__ P, const CpqrChunk* __restrict__ chunks,
                                                   int nchunk, int t, int* __restrict__ counter) {
  __shared__ int s_ci, s_last;
  for (;;) {
    if (threadIdx.x == 0) s_ci = atomicAdd(counter, 1);
    __syncthreads();
    const int ci = s_ci;
    if (ci >= nchunk) break;
    const CpqrChunk ch = chunks[ci];
    const CpqrProb<C> p = P[ch.id];
    const int s = p.base + t;
    // the matrix's pick is rewritten only after all of its chunks are done
    const CpqrPick<C> pk = *p.pick;
    if (s < p.target && pk.q >= 0) {
      if constexpr (sizeof(C) == 16) cpqr_columns_fx(p, ch, s, pk);
      else cpqr_columns<C, TALL>(p, ch, s, pk);
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) {
        s_last = atomicAdd(p.done, 1) == (p.n + CPQR_CB - 1) / CPQR_CB - 1;
        if (s_last) *p.done = 0;
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        cpqr_pick<C>(p, s + 1);
      }
    }
    __syncthreads();
  }
}

// ---- all steps of a small matrix in one launch ------------------------------------------
// A matrix whose columns fit the shared memory of a cluster (up to 8 CTAs) runs
// its whole phase there: column c in CTA c % cs, a warp per column.  Per step
// one cluster barrier, after which every CTA reads all norms and the pivot
// column from the others' shared memory and forms the same reflector: a few
// microseconds, against a launch, a chunk's descriptors and the L2 round trips
// of k_cpqr_step (20 us and more however small the matrix).  Per column the
// arithmetic is that of k_cpqr_step; in complex128 the sums are exact, so the
// bits are the same too.
constexpr int RT = 512;
constexpr int RES_MAX_N = 512;      // a thread per column when the norms are compared
constexpr int RES_MAX_COLS = 192;   // local columns
constexpr size_t RES_SMEM = 200 * 1024;

template <typename C>
__global__ void __launch_bounds__(RT, 1) k_cpqr_resident(const CpqrProb<C>* __restrict__ P, const int* __restrict__ list) {
  namespace cg = cooperative_groups;
  typedef typename real_of<C>::type R;
  typedef unsigned long long u64;
  constexpr bool FX = sizeof(C) == 16;
  constexpr int NW = RT / 32;
  extern __shared__ __align__(16) unsigned char rs_sm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const CpqrProb<C> p = P[list[blockIdx.x / cs]];
  const int n = p.n, W = p.W, ncl = n > rank ? (n - rank + cs - 1) / cs : 0;   // this CTA's columns rank, rank + cs, ..
  C* s_x = reinterpret_cast<C*>(rs_sm);                  // the pivot column (complex128: shifted integers)
  C* s_c = s_x + W;                                      // columns, leading dimension W
  __shared__ double s_norm[2][RES_MAX_COLS];             // trailing norms by step parity (-1: pivoted)
  __shared__ u64 s_k[NW];
  __shared__ int s_i[NW];
  __shared__ C s_ctau, s_csc, s_sc;
  __shared__ int s_ev;
  __shared__ longlong2 s_dot[FX ? RES_MAX_COLS : 1], s_nrm[FX ? RES_MAX_COLS : 1];
  __shared__ uint2 s_dlo[FX ? RES_MAX_COLS : 1];
  __shared__ int4 s_g[FX ? RES_MAX_COLS : 1];
  __shared__ int2 s_gn[FX ? RES_MAX_COLS : 1];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int l = warp; l < ncl; l += NW) {
    const C* src = p.Z + (size_t)(rank + cs * l) * p.ld;
    for (int r = lane; r < W; r += 32) s_c[(size_t)l * W + r] = src[r];
  }
  for (int l = tid; l < ncl; l += RT) s_norm[p.base & 1][l] = p.norm2[(p.base & 1) * n + rank + cs * l];
  double ref = p.mode == CPQR_FIND_RANK && p.base > 0 ? *p.ref : 0.0;
  int s = p.base;
  for (; s < p.target; ++s) {
    const int par = s & 1;
    cluster.sync();   // the norms of step s are complete everywhere
    // the largest norm, then the lowest column within the tie band
    u64 key = 0;
    if (tid < n) {
      const u64 b = (u64)__double_as_longlong(cluster.map_shared_rank(&s_norm[par][0], tid % cs)[tid / cs]);
      key = b <= 0x7FF0000000000000ull ? b + 1 : 0;   // 0: pivoted or not a number
    }
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(key >> 32) == hi ? (unsigned)key : 0u);
    if (lane == 0) s_k[warp] = ((u64)hi << 32) | lo;
    __syncthreads();
    u64 k = s_k[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) k = s_k[w] > k ? s_k[w] : k;
    const double mx = k ? __longlong_as_double((long long)(k - 1)) : 0.0;
    const u64 band = k ? (u64)__double_as_longlong((1.0 - TIE) * mx) + 1 : ~0ull;
    const int qw = __reduce_min_sync(0xffffffffu, key >= band ? tid : RES_MAX_N);
    if (lane == 0) s_i[warp] = qw;
    __syncthreads();
    int q = s_i[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) q = min(q, s_i[w]);
    if (!k || q >= n) break;   // no unpivoted column left (the same in every CTA)
    if (p.mode == CPQR_FIND_RANK) {
      if (s == 0) {
        ref = sqrt(mx);
        if (rank == 0 && tid == 0) *p.ref = ref;
      }
      if (!(sqrt(mx) > p.tol * ref)) {
        if (rank == 0 && tid == 0) *p.rank = s;
        break;
      }
    }
    const int qr = q % cs, ql = q / cs;
    const double nq = cluster.map_shared_rank(&s_norm[par][0], qr)[ql];
    const C* xq = cluster.map_shared_rank(s_c, qr) + (size_t)ql * W;
    int ev = 0;
    if constexpr (FX) {
      const int eq = p.cexp[q];
      const double nn = ldexp(nq, -2 * eq);   // in units of the column's scale
      ev = fx_shift(nq, eq);
      for (int r = s + 1 + tid; r < W; r += RT) {
        const longlong2 v = *reinterpret_cast<const longlong2*>(xq + r);
        *reinterpret_cast<longlong2*>(s_x + r) = make_longlong2(v.x << ev, v.y << ev);
      }
      if (warp == NW - 1) {
        const longlong2 a = *reinterpret_cast<const longlong2*>(xq + s);
        double beta;
        double2 tau, sc;
        fx_reflector(make_double2(fx_to(a.x, 0), fx_to(a.y, 0)), nn, beta, tau, sc);
        if (lane == 0) {
          s_ctau = conj(tau);
          s_sc = __longlong_as_double((long long)(1023 - ev) << 52) * sc;
          s_csc = __longlong_as_double((long long)(1023 - 60 - ev) << 52) * conj(sc);
          if (rank == 0) {
            p.rdiag[s] = make_double2(ldexp(beta != 0 ? beta : 0x1p-58, eq), 0.0);
            p.perm[s] = q;
          }
        }
      }
    } else {
      for (int r = s + 1 + tid; r < W; r += RT) s_x[r] = xq[r];
      if (warp == NW - 1) {
        const C alpha = xq[s];
        const R xnorm = (R)sqrt(nq);
        const R beta = -copysign(xnorm, alpha.x);
        C tau = czero<C>(), sc = czero<C>();
        if (xnorm > 0) {
          const C bm = mk(beta, (R)0);
          tau = cdiv(bm - alpha, bm);
          sc = cdiv(mk((R)1, (R)0), alpha - bm);
        }
        if (lane == 0) {
          s_ctau = conj(tau);
          s_sc = sc;
          s_csc = conj(sc);
          if (rank == 0) {
            p.rdiag[s] = mk(beta, (R)0);
            p.perm[s] = q;
          }
        }
      }
    }
    __syncthreads();
    auto active = [&](int l) { return !(s_norm[par][l] < 0) && rank + cs * l != q; };
    if constexpr (FX) {
      const longlong2* x = reinterpret_cast<const longlong2*>(s_x);
      for (int l = warp; l < ncl; l += NW) {
        if (!active(l)) continue;
        const longlong2* a = reinterpret_cast<const longlong2*>(s_c + (size_t)l * W);
        const int ea = fx_shift(s_norm[par][l], p.cexp[rank + cs * l]);
        longlong2 d = make_longlong2(0, 0);
        for (int r = s + 1 + lane; r < W; r += 32) fx_dot(d, x[r], a[r], ea);
        longlong2 h;
        uint2 lw;
        warp_sum_parts(d.x, h.x, lw.x);
        warp_sum_parts(d.y, h.y, lw.y);
        if (lane == 0) { s_dot[l] = h; s_dlo[l] = lw; }
      }
      __syncthreads();
      for (int l = tid; l < ncl; l += RT)
        if (active(l))
          fx_factor(s_ctau, s_csc, s_sc, s_dot[l], s_dlo[l], fx_shift(s_norm[par][l], p.cexp[rank + cs * l]),
                    reinterpret_cast<longlong2*>(s_c + (size_t)l * W + s), s_g[l], s_gn[l]);
      __syncthreads();
      for (int l = warp; l < ncl; l += NW) {
        if (!active(l)) continue;
        longlong2* a = reinterpret_cast<longlong2*>(s_c + (size_t)l * W);
        const int4 g = s_g[l];
        const int2 gn = s_gn[l];
        FxSquares sq;
        int it = 0;
        for (int r = s + 1 + lane; r < W; r += 32) {
          a[r] = fx_update(a[r], x[r], g, gn);
          sq.add(a[r]);
          if ((++it & 7) == 0) sq.fold();
        }
        const longlong2 w = sq.warp_total();
        if (lane == 0) s_nrm[l] = w;
      }
      __syncthreads();
      for (int l = tid; l < ncl; l += RT)
        s_norm[par ^ 1][l] = active(l) ? fx_norm2(s_nrm[l], p.cexp[rank + cs * l]) : -1.0;
    } else {
      const C ctau = s_ctau, sc = s_sc, csc = s_csc;
      for (int l = warp; l < ncl; l += NW) {
        if (!active(l)) {
          if (lane == 0) s_norm[par ^ 1][l] = -1.0;
          continue;
        }
        C* a = s_c + (size_t)l * W;
        C dot = czero<C>();
        for (int r = s + 1 + lane; r < W; r += 32) cfma_conj(dot, s_x[r], a[r]);
        dot.x = warp_sum(dot.x);
        dot.y = warp_sum(dot.y);
        const C a_s = a[s];
        __syncwarp();
        const C f = ctau * (a_s + csc * dot), fs = f * sc;   // as in cpqr_columns
        if (lane == 0) a[s] = a_s - f;
        R e = 0;
        for (int r = s + 1 + lane; r < W; r += 32) {
          C v = a[r];
          cfms(v, fs, s_x[r]);
          a[r] = v;
          e += abs2(v);
        }
        e = warp_sum(e);
        if (lane == 0) s_norm[par ^ 1][l] = (double)e;
      }
    }
  }
  cluster.sync();   // no CTA leaves while another may still read its norms or columns
  // the norms of step s and the columns, for a later phase
  for (int l = tid; l < ncl; l += RT) p.norm2[(s & 1) * n + rank + cs * l] = s_norm[s & 1][l];
  for (int l = warp; l < ncl; l += NW) {
    C* dst = p.Z + (size_t)(rank + cs * l) * p.ld;
    for (int r = lane; r < W; r += 32) dst[r] = s_c[(size_t)l * W + r];
  }
}

// R11 (k x k, upper, diagonal from rdiag, zero below) and R12 (into T) in
// pivot order, both with leading dimension k.
template <typename C>
__global__ void k_interp_gather(const InterpProb<C>* __restrict__ P) {
  const InterpProb<C> p = P[blockIdx.y];
  const int k = p.k;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k <= 0 || e >= (size_t)k * p.n) return;
  const int i = (int)(e % k), j = (int)(e / k);
  C v = p.Z[i + (size_t)p.perm[j] * p.ld];
  if constexpr (sizeof(C) == 16) {   // complex128 columns are in fixed point
    const int e = p.cexp[p.perm[j]];
    v = make_double2(fx_to(__double_as_longlong(v.x), e), fx_to(__double_as_longlong(v.y), e));
  }
  if (j < k) p.R11[i + (size_t)j * k] = i < j ? v : (i == j ? p.rdiag[i] : czero<C>());
  else p.T[i + (size_t)(j - k) * p.ldt] = v;
}

template <typename C>
__global__ void k_scatter(const ScatterProb<C>* __restrict__ P) {
  typedef typename real_of<C>::type R;
  const ScatterProb<C> p = P[blockIdx.y];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= p.k * p.ng) return;
  const int j = e % p.k, c = e / p.k;
  C v;
  if (c < p.k) {
    if (c != j) return;
    v = mk((R)1, (R)0);
  } else {
    v = p.T[j + (size_t)(c - p.k) * p.ldt];
  }
  const int row = p.pos[p.perm[c]];
  if (p.isL) p.out[row + (size_t)(p.off + j) * p.ld] = v;
  else p.out[(p.off + j) + (size_t)row * p.ld] = v;
}

__device__ __forceinline__ double2 cvt(double2 a, double2*) { return a; }
__device__ __forceinline__ float2 cvt(float2 a, float2*) { return a; }
__device__ __forceinline__ double2 cvt(float2 a, double2*) { return make_double2(a.x, a.y); }
__device__ __forceinline__ float2 cvt(double2 a, float2*) { return make_float2((float)a.x, (float)a.y); }

template <typename S, typename D>
__global__ void k_copy(const CopyProb<S, D>* __restrict__ P) {
  const CopyProb<S, D> p = P[blockIdx.y];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= p.m * p.n) return;
  const int i = e % p.m, j = e / p.m;
  p.dst[i + (size_t)j * p.ldd] = cvt(p.src[i + (size_t)j * p.lds], (D*)nullptr);
}

// Completes a permutation: after `done` pivot steps, the remaining columns in
// ascending order (one CTA per matrix).
__global__ void k_complete_perm(const PermFill* __restrict__ P) {
  extern __shared__ unsigned char used[];
  const PermFill p = P[blockIdx.x];
  for (int c = threadIdx.x; c < p.n; c += blockDim.x) used[c] = 0;
  __syncthreads();
  for (int s = threadIdx.x; s < p.done; s += blockDim.x) used[p.perm[s]] = 1;
  __syncthreads();
  if (threadIdx.x == 0) {
    int o = p.done;
    for (int c = 0; c < p.n; ++c) if (!used[c]) p.perm[o++] = c;
  }
}

}  // namespace

void complete_perm(const PermFill* d_prob, int nprob, cudaStream_t st) {
  if (nprob <= 0) return;
  static std::once_flag attr;
  std::call_once(attr, [] { cudaFuncSetAttribute(k_complete_perm, cudaFuncAttributeMaxDynamicSharedMemorySize, 65536); });
  k_complete_perm<<<nprob, 256, 65536, st>>>(d_prob);
  pm_launch_count_add(1);
}

template <typename C>
void cpqr_init_norms(const CpqrProb<C>* d_prob, const CpqrChunk* d_chunk, int nchunk, cudaStream_t st) {
  if (nchunk <= 0) return;
  k_init_norms<C><<<nchunk, 256, 0, st>>>(d_prob, d_chunk);
  pm_launch_count_add(1);
}
template <typename C>
void cpqr_start(const CpqrProb<C>* d_prob, int nprob, cudaStream_t st) {
  if (nprob <= 0) return;
  k_cpqr_start<C><<<nprob, 256, 0, st>>>(d_prob);
  pm_launch_count_add(1);
}
template <typename C>
int cpqr_resident_ctas(int n, int W) {
  for (int cs = 1; cs <= 8; cs *= 2) {
    const size_t cols = (n + cs - 1) / cs;
    if (n <= RES_MAX_N && cols <= RES_MAX_COLS && (cols + 1) * W * sizeof(C) <= RES_SMEM) return cs;
  }
  return 0;
}
template <typename C>
void cpqr_resident(const CpqrProb<C>* d_prob, const int* d_list, const int* h_n, const int* h_w, int count, int cs,
                   int sms, cudaStream_t st) {
  if (count <= 0) return;
  const int max_n = *std::max_element(h_n, h_n + count);
  while (cs < 8 && (long)count * cs * 2 <= sms && cs * 32 <= max_n) cs *= 2;   // spread a few matrices wider
  size_t bytes = 0;
  for (int i = 0; i < count; ++i) bytes = std::max(bytes, ((size_t)(h_n[i] + cs - 1) / cs + 1) * h_w[i] * sizeof(C));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(count * cs);
  cfg.blockDim = dim3(RT);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // the same value every time: idempotent across threads and devices
  cudaFuncSetAttribute(k_cpqr_resident<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RES_SMEM);
  KPROF_BEGIN(st);
  cudaLaunchKernelEx(&cfg, k_cpqr_resident<C>, d_prob, d_list);
  pm_launch_count_add(1);
  KPROF_END(st, kname<C>("cpqr_resident", "cpqr_resident32"), 0.0);
}
template <typename C, bool TALL>
int cpqr_grid() {   // SMs x resident CTAs, once per instance
  static std::atomic<int> grid_cache{0};
  int grid = grid_cache.load();
  if (grid == 0) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cpqr_step<C, TALL>, 256, 0);
    grid = std::max(1, sms * std::max(per, 1));
    grid_cache.store(grid);
  }
  return grid;
}

template <typename C>
void cpqr_step(const CpqrProb<C>* d_prob, const CpqrChunk* d_chunk, int nchunk, int t, int* d_counter,
               cudaStream_t st, bool tall) {
  if (nchunk <= 0) return;
  KPROF_BEGIN(st);
  if (tall && sizeof(C) == 8) k_cpqr_step<C, true><<<std::min(cpqr_grid<C, true>(), nchunk), 256, 0, st>>>(d_prob, d_chunk, nchunk, t, d_counter);
  else k_cpqr_step<C, false><<<std::min(cpqr_grid<C, false>(), nchunk), 256, 0, st>>>(d_prob, d_chunk, nchunk, t, d_counter);
  pm_launch_count_add(1);
  KPROF_END(st, kname<C>("cpqr_step", "cpqr_step32"), 0.0);   // work is added per level from the steps performed
}
template <typename C>
void interp_gather(const InterpProb<C>* d_prob, int nprob, size_t max_elems, cudaStream_t st) {
  if (nprob <= 0 || max_elems == 0) return;
  dim3 g((unsigned)((max_elems + 255) / 256), nprob);
  k_interp_gather<C><<<g, 256, 0, st>>>(d_prob);
  pm_launch_count_add(1);
}
template <typename C>
void scatter_interp(const ScatterProb<C>* d_prob, int nprob, int max_elems, cudaStream_t st) {
  if (nprob <= 0 || max_elems <= 0) return;
  dim3 g((max_elems + 255) / 256, nprob);
  k_scatter<C><<<g, 256, 0, st>>>(d_prob);
  pm_launch_count_add(1);
}
template <typename S, typename D>
void copy_batched(const CopyProb<S, D>* d_prob, int nprob, int max_elems, cudaStream_t st) {
  if (nprob <= 0 || max_elems <= 0) return;
  dim3 g((max_elems + 255) / 256, nprob);
  k_copy<S, D><<<g, 256, 0, st>>>(d_prob);
  pm_launch_count_add(1);
}

template void cpqr_init_norms<double2>(const CpqrProb<double2>*, const CpqrChunk*, int, cudaStream_t);
template int cpqr_resident_ctas<double2>(int, int);
template int cpqr_resident_ctas<float2>(int, int);
template void cpqr_resident<double2>(const CpqrProb<double2>*, const int*, const int*, const int*, int, int, int, cudaStream_t);
template void cpqr_resident<float2>(const CpqrProb<float2>*, const int*, const int*, const int*, int, int, int, cudaStream_t);
template void cpqr_start<double2>(const CpqrProb<double2>*, int, cudaStream_t);
template void cpqr_start<float2>(const CpqrProb<float2>*, int, cudaStream_t);
template void cpqr_step<double2>(const CpqrProb<double2>*, const CpqrChunk*, int, int, int*, cudaStream_t, bool);
template void interp_gather<double2>(const InterpProb<double2>*, int, size_t, cudaStream_t);
template void scatter_interp<double2>(const ScatterProb<double2>*, int, int, cudaStream_t);
template void copy_batched<double2, double2>(const CopyProb<double2, double2>*, int, int, cudaStream_t);
template void copy_batched<float2, float2>(const CopyProb<float2, float2>*, int, int, cudaStream_t);
template void copy_batched<float2, double2>(const CopyProb<float2, double2>*, int, int, cudaStream_t);
template void copy_batched<double2, float2>(const CopyProb<double2, float2>*, int, int, cudaStream_t);
template void cpqr_init_norms<float2>(const CpqrProb<float2>*, const CpqrChunk*, int, cudaStream_t);
template void cpqr_step<float2>(const CpqrProb<float2>*, const CpqrChunk*, int, int, int*, cudaStream_t, bool);
template void interp_gather<float2>(const InterpProb<float2>*, int, size_t, cudaStream_t);
template void scatter_interp<float2>(const ScatterProb<float2>*, int, int, cudaStream_t);
