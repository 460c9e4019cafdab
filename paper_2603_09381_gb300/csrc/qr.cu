// Blocked, unpivoted Householder QR of the tall ID inputs (W x n, W > n),
// ahead of their column-pivoted QR (paper Sec. 3 computes the ID by CPQR).
// Q^H preserves the norm of every trailing column block, so the pivoted
// factorization of the n x n triangle R picks the pivots of Z and returns its
// R (exact arithmetic); the pivoted steps then stream n instead of W rows.
//
// Per panel of QR_NB columns: a cluster of 1-8 CTAs per matrix factors the
// panel (LAPACK zlarfg phase convention, H = I - tau v v^H, Q^H applied) with
// one pass over the panel per reflector (the pass that applies reflector j
// also sums the norm and the dot products that define reflector j+1); the
// cluster's CTAs split the rows and add their partial sums through
// distributed shared memory, every CTA forming the same reflector from the
// same sums.  It then forms the compact-WY factor T (Q = I - V T V^H).
// Q^H = I - V T^H V^H is applied to every 32-column tile of the trailing
// block in three launches: partial products Y_b = V_b^H C_b per (tile,
// QR_RB-row block), their sum in block order times T^H, and C_b -= V_b Y per
// (tile, block), so that the rows of a tall matrix spread over many CTAs.
#include "cpqr.cuh"
#include "fx.cuh"
#include "prof.cuh"
#include "oz.cuh"
#include "oz_gemm.cuh"
#include "tc_common.cuh"
#include <cooperative_groups.h>
#include <type_traits>

namespace cg = cooperative_groups;

namespace {

constexpr int PT = 512;      // panel CTA
constexpr int UT = 256;      // update CTA
constexpr int RC = 32;       // rows per staged chunk
// Q threads share a row of the panel, thread q holding columns q, q + Q, ..
// Interleaved, the columns already factored drop out for all Q threads at
// once: a warp's instructions shrink with the trailing block (a split in
// halves kept every instruction alive until the last column).
template <int Q_> struct PanelSplit {
  static constexpr int Q = Q_;
  static constexpr int HB = QR_NB / Q;      // columns per thread
  static constexpr int RW = 32 / Q;         // rows per warp and sweep
  static constexpr int PR = PT / Q;         // rows per sweep of the CTA
  static_assert(RW == HB, "the reduction below leaves one column per lane");
};

// V entry (row r, panel column j) of a panel starting at j0: unit diagonal,
// zero above, the stored reflector below.
template <typename C>
__device__ __forceinline__ C v_entry(const QrProb<C>& p, int j0, int jb, int r, int j) {
  typedef typename real_of<C>::type R;
  if (j >= jb || r >= p.W) return czero<C>();
  const int d = j0 + j;
  if (r < d) return czero<C>();
  if (r == d) return mk((R)1, (R)0);
  return p.Z[r + (size_t)d * p.ld];
}

__device__ __forceinline__ float2 shfl_xor_c(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ longlong2 shfl_xor_c(longlong2 v, int o) {
  return make_longlong2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// ---- complex64 panel ----------------------------------------------------------------
// A panel of 32 columns in four sub-panels of SB = 8 on a cluster, each CTA
// with a block of rows, a thread per row.  What bounded the plain right-looking
// panel was the L2: every column's pass read and wrote all columns to its
// right (16 of them on average) for one multiply-add per byte.  The 8 columns
// of a sub-panel stay in shared memory (SM; in place, in L2, when a CTA has
// more than SUB_ROWS rows) while their reflectors are found; the columns to
// the right are then updated once per sub-panel, C -= V w with
//   w_j = conj(tau_j) (v_j^H C - sum_{l<j} v_j^H v_l w_l),
// and the products V^H [earlier V, V, C] of that update also give G = V^H V for
// the compact-WY factor T (the sums over rows once per 256 products instead of
// a separate pass).  Per column one cluster barrier: every CTA pushes its
// partial sums to the others before it, and every warp forms the reflector
// (LAPACK zlarfg phase) from them.
// At most 112 registers: 512 x 112 leaves room on the SM for one CTA of the
// operator assembly that may run beside the factorization.
constexpr int SB = 8;
constexpr int SUB_ROWS = 2560;                                    // x 64 bytes: 160 KB
constexpr int YV = QR_NB * SB;                                    // products per sub-panel
constexpr size_t PANEL_RED = (size_t)(PT / 32) * YV * sizeof(float2);   // every warp's
template <bool SM>
__global__ void __maxnreg__(112) k_qr_panel(const QrProb<float2>* __restrict__ P, int j0, int ldp) {
  typedef float2 C;
  cg::cluster_group cluster = cg::this_cluster();
  const int csize = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const QrProb<C> p = P[blockIdx.x / csize];
  if (j0 >= p.n) return;   // the whole cluster (same matrix) leaves
  const int jb = min(QR_NB, p.n - j0), W = p.W;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NS = 2 * SB + 1, NV = NS + 2 * SB;   // S (re, im), N; row c' (re, im)
  extern __shared__ __align__(16) unsigned char qr_sm[];
  C* s_yw = reinterpret_cast<C*>(qr_sm);                       // [PT / 32][YV]
  C (*s_t)[QR_NB + 1] = reinterpret_cast<C (*)[QR_NB + 1]>(qr_sm);   // (after the last sub-panel)
  __shared__ float s_red[PT / 32][NS];
  __shared__ float s_in[2][8][NV];     // the CTAs' partial sums, by pass parity
  __shared__ C s_row[SB];              // row c' (rank 0 has the pivot rows)
  __shared__ C s_tau[QR_NB];
  __shared__ C s_y[YV], s_yt[YV];      // V^H [..]: this CTA's, the cluster's ([column][l])
  __shared__ C s_w[QR_NB][SB];
  __shared__ C s_g[QR_NB][QR_NB + 1];  // s_g[j][l] = v_j^H v_l, l <= j
  // block of rows, a multiple of 32 (so rank 0 holds all pivot rows)
  const int nr = ((W - j0 + csize - 1) / csize + 31) & ~31, rb = j0 + rank * nr, re = min(W, rb + nr);
  const size_t ld = p.ld;
  C* Zp = p.Z + (size_t)j0 * ld;       // panel column k at Zp + k ld
  if (SM) {
    C* X = reinterpret_cast<C*>(qr_sm + PANEL_RED);
    for (int r = rb + tid; r < re; r += PT)
#pragma unroll
      for (int k = 0; k < SB; ++k)
        if (k < jb) X[r - rb + k * ldp] = Zp[r + (size_t)k * ld];
  }
  if (tid < SB) s_row[tid] = make_float2(0.f, 0.f);
  for (int e = tid; e < QR_NB * (QR_NB + 1); e += PT) (&s_g[0][0])[e] = make_float2(0.f, 0.f);
  cluster.sync();   // no CTA writes to one that has not started
  int par = 0;
  for (int c0 = 0; c0 < jb; c0 += SB) {
    const int nb = min(SB, jb - c0);
    C* X = SM ? reinterpret_cast<C*>(qr_sm + PANEL_RED) - rb : Zp + (size_t)c0 * ld;   // row r of column k: X[r + k ldx]
    const size_t ldx = SM ? (size_t)ldp : ld;
    C f[SB], sc = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < SB; ++k) f[k] = make_float2(0.f, 0.f);
    for (int ja = -1; ja < nb; ++ja, par ^= 1) {
      // reflector ja applied (its column scaled into v); for step jn = ja + 1:
      // N = sum_{r >= c'} |a_jn|^2, S_k = sum_{r > c'} conj(a_jn) a_k, k > jn
      const int jn = ja + 1, ca = j0 + c0 + ja, cn = ca + 1;
      float N = 0.f;
      C S[SB];
#pragma unroll
      for (int k = 0; k < SB; ++k) S[k] = make_float2(0.f, 0.f);
      for (int r = rb + tid; r < re; r += PT) {
        if (r < (ja >= 0 ? ca : cn)) continue;
        C a[SB];
#pragma unroll
        for (int k = 0; k < SB; ++k) a[k] = (k > ja && k < nb) ? X[r + k * ldx] : make_float2(0.f, 0.f);
        if (ja >= 0) {
          C v = make_float2(1.f, 0.f);
          if (r > ca) {
            v = X[r + ja * ldx] * sc;
            X[r + ja * ldx] = v;
          }
#pragma unroll
          for (int k = 0; k < SB; ++k)
            if (k > ja && k < nb) {
              cfms(a[k], f[k], v);
              X[r + k * ldx] = a[k];
            }
        }
        if (jn < nb && r >= cn) {
          C y = a[0];
#pragma unroll
          for (int k = 1; k < SB; ++k)
            if (k == jn) y = a[k];
          N += abs2(y);
          if (r == cn) {
#pragma unroll
            for (int k = 0; k < SB; ++k) s_row[k] = a[k];
          } else {
#pragma unroll
            for (int k = 0; k < SB; ++k)
              if (k > jn) cfma_conj(S[k], y, a[k]);
          }
        }
      }
      if (jn >= nb) break;
      // warp sums, halving the columns with the first exchanges: column lane / 4
      N = warp_sum(N);
#pragma unroll
      for (int o = 16, cnt = SB / 2; o >= 4; o >>= 1, cnt >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < SB / 2; ++k)
          if (k < cnt) {
            const C send = up ? S[k] : S[k + cnt], keep = up ? S[k + cnt] : S[k];
            S[k] = keep + shfl_xor_c(send, o);
          }
      }
      S[0] = S[0] + shfl_xor_c(S[0], 2);
      S[0] = S[0] + shfl_xor_c(S[0], 1);
      if ((lane & 3) == 0) {
        s_red[warp][lane >> 1] = S[0].x;
        s_red[warp][(lane >> 1) + 1] = S[0].y;
      }
      if (lane == 0) s_red[warp][2 * SB] = N;
      __syncthreads();
      for (int t = tid; t < csize * NV; t += PT) {
        const int dst = t / NV, i = t % NV;
        float u = 0.f;
        if (i < NS) {
#pragma unroll
          for (int w = 0; w < PT / 32; ++w) u += s_red[w][i];
        } else {
          u = reinterpret_cast<const float*>(s_row)[i - NS];
        }
        cluster.map_shared_rank(&s_in[par][rank][0], dst)[i] = u;
      }
      cluster.sync();   // every CTA's partials of this pass have arrived
      // lanes 0 .. 15: S, 16 .. 31: row c'; N in all
      float t = lane < 2 * SB ? 0.f : s_in[par][0][lane + 1];
      N = 0.f;
      for (int r = 0; r < csize; ++r) {   // rank order
        if (lane < 2 * SB) t += s_in[par][r][lane];
        N += s_in[par][r][2 * SB];
      }
      const C alpha = make_float2(__shfl_sync(0xffffffffu, t, 2 * SB + 2 * jn), __shfl_sync(0xffffffffu, t, 2 * SB + 2 * jn + 1));
      const int kk = lane & (SB - 1);
      const C Sk = make_float2(__shfl_sync(0xffffffffu, t, 2 * kk), __shfl_sync(0xffffffffu, t, 2 * kk + 1));
      const C rowk = make_float2(__shfl_sync(0xffffffffu, t, 2 * SB + 2 * kk), __shfl_sync(0xffffffffu, t, 2 * SB + 2 * kk + 1));
      const float xnorm = sqrtf(N);
      C tau = make_float2(0.f, 0.f);
      float beta = 0.f;
      sc = tau;
      if (xnorm > 0.f) {
        beta = -copysignf(xnorm, alpha.x);
        const C bm = make_float2(beta, 0.f);
        tau = cdiv(bm - alpha, bm);
        sc = cdiv(make_float2(1.f, 0.f), alpha - bm);
      }
      const C fk = conj(tau) * (rowk + conj(sc) * Sk);
#pragma unroll
      for (int k = 0; k < SB; ++k)
        f[k] = make_float2(__shfl_sync(0xffffffffu, fk.x, k), __shfl_sync(0xffffffffu, fk.y, k));
      if (rank == 0 && cn < re && tid == (cn - rb) % PT) X[cn + jn * ldx] = make_float2(beta, 0.f);   // (the row's thread)
      if (tid == 0) s_tau[c0 + jn] = tau;
    }
    // V^H [earlier V, V, C], 4 columns at a time
    auto masked = [&](C x, int r, int col) {
      const int e = r - (j0 + col);
      return e > 0 ? x : make_float2(e == 0 ? 1.f : 0.f, 0.f);
    };
    auto v_row = [&](int r, C* v) {
#pragma unroll
      for (int l = 0; l < SB; ++l) v[l] = l < nb ? X[r + l * ldx] : make_float2(0.f, 0.f);
      if (r < j0 + QR_NB) {
#pragma unroll
        for (int l = 0; l < SB; ++l) v[l] = l < nb ? masked(v[l], r, c0 + l) : make_float2(0.f, 0.f);
      }
    };
    for (int k0 = 0; k0 < QR_NB; k0 += 4) {
      C acc[4 * SB];
#pragma unroll
      for (int i = 0; i < 4 * SB; ++i) acc[i] = make_float2(0.f, 0.f);
      if (k0 < jb) {
        const bool own = k0 >= c0 && k0 < c0 + SB;
        const C* src = own ? X + (size_t)(k0 - c0) * ldx : Zp + (size_t)k0 * ld;
        const size_t lds = own ? ldx : ld;
        for (int r = rb + tid; r < re; r += PT) {
          C v[SB], c[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) c[i] = k0 + i < jb ? src[r + i * lds] : make_float2(0.f, 0.f);
          if (r < j0 + QR_NB && k0 < c0 + SB) {
#pragma unroll
            for (int i = 0; i < 4; ++i) c[i] = k0 + i < jb ? masked(c[i], r, k0 + i) : make_float2(0.f, 0.f);
          }
          v_row(r, v);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int l = 0; l < SB; ++l) cfma_conj(acc[i * SB + l], v[l], c[i]);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {   // lane i ends with product i
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < 2 * SB; ++k)
          if (k < o) {
            const C send = up ? acc[k] : acc[k + o], keep = up ? acc[k + o] : acc[k];
            acc[k] = keep + shfl_xor_c(send, o);
          }
      }
      s_yw[warp * YV + k0 * SB + lane] = acc[0];
    }
    __syncthreads();
    {
      float u = 0.f;
#pragma unroll
      for (int w = 0; w < PT / 32; ++w) u += reinterpret_cast<const float*>(s_yw)[w * 2 * YV + tid];
      reinterpret_cast<float*>(s_y)[tid] = u;
    }
    cluster.sync();
    {
      float u = 0.f;
      for (int r = 0; r < csize; ++r) u += reinterpret_cast<const float*>(cluster.map_shared_rank(&s_y[0], r))[tid];   // rank order
      reinterpret_cast<float*>(s_yt)[tid] = u;
    }
    __syncthreads();
    if (warp == 0) {
      const int k = lane;
      C w[SB];
#pragma unroll
      for (int j = 0; j < SB; ++j) {
        C y = s_yt[k * SB + j];
        if (j < nb && k <= c0 + j) s_g[c0 + j][k] = y;
#pragma unroll
        for (int l = 0; l < j; ++l) cfms(y, s_yt[(c0 + l) * SB + j], w[l]);
        w[j] = j < nb ? conj(s_tau[c0 + j]) * y : make_float2(0.f, 0.f);
        s_w[k][j] = w[j];
      }
    }
    __syncthreads();
    for (int r = rb + tid; r < re; r += PT) {
      C v[SB];
      if (SM) {
#pragma unroll
        for (int l = 0; l < SB; ++l)
          if (l < nb) Zp[r + (size_t)(c0 + l) * ld] = X[r + l * ldx];
      }
      v_row(r, v);
      if (p.V) {
#pragma unroll
        for (int l = 0; l < SB; ++l) p.V[(r - j0) + (size_t)(c0 + l) * W] = v[l];
      }
#pragma unroll 4
      for (int k = c0 + SB; k < jb; ++k) {
        C c = Zp[r + (size_t)k * ld];
#pragma unroll
        for (int l = 0; l < SB; ++l) cfms(c, v[l], s_w[k][l]);
        if (SM && k < c0 + 2 * SB) X[r + (k - c0 - SB) * ldx] = c;
        else Zp[r + (size_t)k * ld] = c;
      }
    }
  }
  if (p.V)
    for (int j = (jb + SB - 1) / SB * SB; j < QR_NB; ++j)
      for (int r = rb + tid; r < re; r += PT) p.V[(r - j0) + (size_t)j * W] = make_float2(0.f, 0.f);
  // T: T_jj = tau_j, T[0:j, j] = -tau_j T[0:j, 0:j] G[0:j, j]; 16 lanes per row
  if (rank == 0) {
    const int i = tid >> 4, part = tid & 15;
    for (int e = tid; e < QR_NB * QR_NB; e += PT) {
      const int a = e % QR_NB, b = e / QR_NB;
      s_t[a][b] = (a == b && a < jb) ? s_tau[a] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int j = 1; j < jb; ++j) {
      C acc = make_float2(0.f, 0.f);
      if (i < j)
        for (int l = i + part; l < j; l += 16) cfma(acc, s_t[i][l], conj(s_g[j][l]));
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) acc = acc + shfl_xor_c(acc, o);
      if (i < j && part == 0) s_t[i][j] = -(s_tau[j] * acc);
      __syncthreads();
    }
    for (int e = tid; e < QR_NB * QR_NB; e += PT) p.T[e] = s_t[e % QR_NB][e / QR_NB];
  }
  cluster.sync();   // no CTA leaves while another may still read its sums
}

// ---- complex128 panel in 60-bit fixed point ----------------------------------------
// The FP64 pipe does 2 fused multiply-adds per clock and SM, the integer
// multipliers 64: a fixed-point complex multiply-add (12 wide multiplies,
// ~10 other instructions) takes a quarter of the time of the 4 FP64 ones.
// Fixed point suits a Householder panel: a reflection keeps the norm of
// a column, so with a scale per column (its norm at most 1/4, a power of two)
// nothing overflows, and every operation errs by ~2^-59 of the column's
// scale, where FP64 errs by 2^-53 of the entry.
//   entries   A = a 2^-60 scale_k, |a|_2 <= 1/4 per column (64-bit integers, in place of the doubles)
//   v         |v| <= 1, 2^-60
//   y         the column that defines the next reflector.  Its norm may be
//             far below its scale, and the reflector must be orthogonal to
//             working precision, so each warp shifts its rows of y up to use
//             all bits before the dot products; the shifts are taken out when
//             the warps' sums meet, in integers as well.
// (fx.cuh holds the arithmetic.)
// A matrix's panel on a cluster; rows go to warps 8 at a time and stay there
// for the whole panel.  T receives the taus.  Same reflectors and order as
// k_qr_panel (LAPACK zlarfg phase convention).
// Four threads per row: their 8 entries and 8 sums fit the registers.
// SM: a CTA's rows (at most FX_SWEEPS per warp and thread) stay in dynamic
// shared memory, leading dimension ldp; else in place, in L2.
constexpr int FX_SWEEPS = 3;   // 3 x 128 rows x 32 columns: 192 KB
template <bool SM>
__global__ void __launch_bounds__(PT, 1) k_qr_panel_fx(const QrProb<double2>* __restrict__ P, int j0, int ldp) {
  typedef PanelSplit<4> L;
  constexpr int Q = L::Q, HB = L::HB, RW = L::RW;
  cg::cluster_group cluster = cg::this_cluster();
  const int csize = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const QrProb<double2> p = P[blockIdx.x / csize];
  if (j0 >= p.n) return;   // the whole cluster (same matrix) leaves
  const int jb = min(QR_NB, p.n - j0), W = p.W;
  extern __shared__ __align__(16) unsigned char fx_sm[];
  const size_t ld = p.ld;
  // the panel's columns as integers: row r, sweep by sweep, at stored row x
  longlong2* Zx = SM ? reinterpret_cast<longlong2*>(fx_sm) : reinterpret_cast<longlong2*>(p.Z + (size_t)j0 * ld);
  const size_t ldx = SM ? ldp : ld;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, q = lane / RW;
  const int rbeg = j0 + warp * RW + rank * L::PR, rstep = L::PR * csize;   // the warp's first row and stride
  const int xbeg = SM ? warp * RW + lane % RW : rbeg + lane % RW, xstep = SM ? L::PR : rstep;
  constexpr int NS = 2 * QR_NB + 2;   // S (re, im), N (low, high)
  __shared__ long long s_red[PT / 32][2 * QR_NB + 1];
  __shared__ int s_ew[PT / 32];
  __shared__ long long s_in[2][8][NS];      // the CTAs' partial sums, by pass parity,
  __shared__ int s_m[2][8];                 // their shifts,
  __shared__ longlong2 s_rowin[2][QR_NB];   // and row c'
  __shared__ double s_nrm[PT / 32][QR_NB], s_n2[QR_NB];
  __shared__ longlong2 s_row[QR_NB];  // row c' (rank 0 has the pivot rows)
  __shared__ int4 s_g[QR_NB];         // factors of the next pass: re, im as (h, l) ..
  __shared__ int2 s_gn[QR_NB];        // .. and -im
  __shared__ long long s_beta[QR_NB]; // R's diagonal: 2^(s_bev - 60) in units of the column's scale
  __shared__ int s_bev[QR_NB];
  __shared__ int s_exp[QR_NB];        // scale of column k: 2^s_exp
  __shared__ int s_bad;               // columns from here on are not finite, or follow one that is not
  __shared__ longlong2 s_tau[QR_NB];  // tau / 2
  __shared__ longlong2 s_sc;
  __shared__ int s_ev;
  // column norms: the scale of column k is the power of two that brings its norm into (1/8, 1/4]
  {
    double acc[HB];
#pragma unroll
    for (int k = 0; k < HB; ++k) acc[k] = 0.0;
    for (int r = rbeg + lane % RW; r < W; r += rstep)
#pragma unroll
      for (int k = 0; k < HB; ++k)
        if (Q * k + q < jb) acc[k] += abs2(p.Z[r + (size_t)(j0 + Q * k + q) * ld]);
#pragma unroll
    for (int k = 0; k < HB; ++k)
#pragma unroll
      for (int o = RW / 2; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (lane % RW == 0)
#pragma unroll
      for (int k = 0; k < HB; ++k) s_nrm[warp][Q * k + q] = acc[k];
    if (tid == 0) s_bad = QR_NB;
    __syncthreads();
    if (tid < QR_NB) {
      double t = 0;
#pragma unroll
      for (int w = 0; w < PT / 32; ++w) t += s_nrm[w][tid];
      s_n2[tid] = t;
    }
    cluster.sync();
    if (tid < jb) {
      double t = 0;
      for (int r = 0; r < csize; ++r) t += cluster.map_shared_rank(&s_n2[0], r)[tid];
      int e = 0;
      if (!isfinite(t)) atomicMin(&s_bad, tid);
      else if (t > 0) frexp(sqrt(t) * (1.0 + 1e-9), &e);
      s_exp[tid] = e + 2;
    }
    __syncthreads();
    for (int r = rbeg + lane % RW, x = xbeg; r < W; r += rstep, x += xstep)
#pragma unroll
      for (int k = 0; k < HB; ++k)
        if (Q * k + q < jb) {
          const double2 z = p.Z[r + (size_t)(j0 + Q * k + q) * ld];
          const int e2 = s_exp[Q * k + q];
          const bool ok = Q * k + q < s_bad;
          Zx[x + (size_t)(Q * k + q) * ldx] = make_longlong2(ok ? fx_from(z.x, e2) : 0, ok ? fx_from(z.y, e2) : 0);
        }
    __syncwarp();
  }
  int par = 0;
  // a row of y is below 2^55 (2^-5) after a warp's shift, less for very tall
  // panels: |S| <= 2^-5 sqrt(2 W) / 4 stays below 2, a warp's N below 1
  const int ytop = 54 - (33 - __clz(W >> 15)) / 2;
  for (int ja = -1; ja < jb; ++ja, par ^= 1) {
    const int jn = ja + 1, ca = j0 + ja, cn = j0 + jn;
    // column ja becomes v, column jn is brought up to date and measured
    Fx scr = {0, 0}, sci = {0, 0}, nsci = {0, 0};
    int ev = 0;
    if (ja >= 0) {
      const longlong2 sc = s_sc;
      scr = fw(sc.x << 2); sci = fw(sc.y << 2); nsci = fw(-sc.y << 2);
      ev = s_ev;
    }
    unsigned long long any = 0;
    // (a thread per row here: the four threads of a row take four sweeps at a time)
    for (int r = rbeg + lane % RW + q * rstep, xr = xbeg + q * xstep; r < W; r += Q * rstep, xr += Q * xstep) {
      if (r < (ja >= 0 ? ca : cn)) continue;
      longlong2 y = jn < jb ? Zx[xr + (size_t)jn * ldx] : make_longlong2(0, 0);
      if (ja >= 0) {
        longlong2 v;
        if (r == ca) {
          v = make_longlong2(1ll << 60, 0);
        } else {
          const longlong2 x = Zx[xr + (size_t)ja * ldx];
          v = fw_cfma(make_longlong2(0, 0), scr, sci, nsci, fw(x.x << (ev + 2)), fw(x.y << (ev + 2)));
          v.x <<= 1; v.y <<= 1;
          Zx[xr + (size_t)ja * ldx] = v;
        }
        if (jn < jb) {
          const int4 g = s_g[jn];
          const int2 gn = s_gn[jn];
          y = fw_cfma(y, Fx{g.x, g.y}, Fx{g.z, g.w}, Fx{gn.x, gn.y}, fw(v.x << 2), fw(v.y << 2));
          Zx[xr + (size_t)jn * ldx] = y;
        }
      }
      if (jn < jb && r >= cn) any |= (unsigned long long)(y.x ^ (y.x >> 63)) | (unsigned long long)(y.y ^ (y.y >> 63));
    }
    __syncwarp();
    if (jn >= jb) break;
    // shift that brings this warp's rows of y just below 2^(ytop + 1)
    const unsigned ah = __reduce_or_sync(0xffffffffu, (unsigned)(any >> 32)), al = __reduce_or_sync(0xffffffffu, (unsigned)any);
    const int top = ah ? 63 - __clz(ah) : (al ? 31 - __clz(al) : 0);
    const int ew = ytop - top;   // top <= 58: may be negative
    long long N = 0;
    longlong2 S[HB];
#pragma unroll
    for (int k = 0; k < HB; ++k) S[k] = make_longlong2(0, 0);
    for (int r = rbeg + lane % RW, xr = xbeg; r < W; r += rstep, xr += xstep) {
      if (r < (ja >= 0 ? ca : cn)) continue;
      longlong2 a[HB];
#pragma unroll
      for (int k = 0; k < HB; ++k)
        if (Q * k + Q - 1 > jn && Q * k + q > jn && Q * k + q < jb) a[k] = Zx[xr + (size_t)(Q * k + q) * ldx];
      const longlong2 v = ja < 0 ? make_longlong2(0, 0) : r == ca ? make_longlong2(1ll << 60, 0) : Zx[xr + (size_t)ja * ldx];
      const longlong2 y0 = Zx[xr + (size_t)jn * ldx];
      // (ew >= -4: the products' 2^4 goes on top)
      const longlong2 y = make_longlong2(y0.x << (ew + 4), y0.y << (ew + 4));
      const Fx vr = fw(v.x << 2), vi = fw(v.y << 2), yr = fw(y.x), yi = fw(y.y), nyi = fw(-y.y);
      if (r >= cn && q == 0) {   // N in 2^-64
        long long cr = FW_HALF;
        fx_mac(N, cr, yr, yr);
        fx_mac(N, cr, yi, yi);
        N += cr >> 32;
      }
      if (r == cn && q == jn % Q) s_row[jn] = y0;
#pragma unroll
      for (int k = 0; k < HB; ++k)
        if (Q * k + Q - 1 > jn && Q * k + q > jn && Q * k + q < jb) {
          if (ja >= 0) {
            const int4 g = s_g[Q * k + q];
            const int2 gn = s_gn[Q * k + q];
            a[k] = fw_cfma(a[k], Fx{g.x, g.y}, Fx{g.z, g.w}, Fx{gn.x, gn.y}, vr, vi);
            Zx[xr + (size_t)(Q * k + q) * ldx] = a[k];
          }
          if (r == cn) {
            s_row[Q * k + q] = a[k];
          } else if (r > cn) {
            const Fx ar = fw(a[k].x), ai = fw(a[k].y);
            long long cr = FW_HALF, ci = FW_HALF;
            fx_mac(S[k].x, cr, yr, ar);
            fx_mac(S[k].x, cr, yi, ai);
            fx_mac(S[k].y, ci, yr, ai);
            fx_mac(S[k].y, ci, nyi, ar);
            S[k].x += cr >> 32;
            S[k].y += ci >> 32;
          }
        }
    }
    __syncwarp();
    // warp sums as in k_qr_panel, in integers
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) N += __shfl_xor_sync(0xffffffffu, N, o);
#pragma unroll
    for (int o = RW / 2, cnt = HB / 2; o > 0; o >>= 1, cnt >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < HB / 2; ++k)
        if (k < cnt) {
          const longlong2 send = up ? S[k] : S[k + cnt], keep = up ? S[k + cnt] : S[k], got = shfl_xor_c(send, o);
          S[k] = make_longlong2(keep.x + got.x, keep.y + got.y);
        }
    }
    {
      const int col = Q * (lane % RW) + q;
      s_red[warp][2 * col] = S[0].x;
      s_red[warp][2 * col + 1] = S[0].y;
      if (lane == 0) { s_red[warp][2 * QR_NB] = N; s_ew[warp] = ew; }
    }
    __syncthreads();
    // over warps, then over CTAs (rank order), each at the smallest shift among
    // them; a CTA pushes its sums to all before the barrier
    if (tid < 2 * QR_NB + 1) {
      int m = s_ew[0];
#pragma unroll
      for (int w = 1; w < PT / 32; ++w) m = min(m, s_ew[w]);
      if (tid < 2 * QR_NB) {
        long long t = 0;
#pragma unroll
        for (int w = 0; w < PT / 32; ++w) t += fx_shr(s_red[w][tid], s_ew[w] - m);
        for (int r = 0; r < csize; ++r) cluster.map_shared_rank(&s_in[par][rank][0], r)[tid] = t;
      } else {
        unsigned __int128 t = 0;
#pragma unroll
        for (int w = 0; w < PT / 32; ++w) t += fx_norm_shr((unsigned __int128)(unsigned long long)s_red[w][tid] << 40, s_ew[w] - m);
        for (int r = 0; r < csize; ++r) {
          long long* dst = cluster.map_shared_rank(&s_in[par][rank][0], r);
          dst[tid] = (long long)t;
          dst[tid + 1] = (long long)(t >> 64);
          *cluster.map_shared_rank(&s_m[par][rank], r) = m;
        }
      }
    } else if (rank == 0 && tid >= 4 * QR_NB && tid < 5 * QR_NB) {
      const longlong2 u = s_row[tid - 4 * QR_NB];
      for (int r = 0; r < csize; ++r) cluster.map_shared_rank(&s_rowin[par][0], r)[tid - 4 * QR_NB] = u;
    }
    cluster.sync();   // every CTA's sums of this pass have arrived
    if (warp == 0) {
      // reflector of column jn, in units of its scale; lane k: the factor of column k
      int M = s_m[par][0];
      for (int r = 1; r < csize; ++r) M = min(M, s_m[par][r]);
      longlong2 Sk = make_longlong2(0, 0);
      unsigned __int128 n2 = 0;
      for (int r = 0; r < csize; ++r) {
        const long long* in = s_in[par][r];
        const int d = s_m[par][r] - M;
        Sk.x += fx_shr(in[2 * lane], d);
        Sk.y += fx_shr(in[2 * lane + 1], d);
        n2 += fx_norm_shr(((unsigned __int128)(unsigned long long)in[2 * QR_NB + 1] << 64) | (unsigned long long)in[2 * QR_NB], d);
      }
      const longlong2 alpha = s_rowin[par][jn];
      int ev;
      longlong2 tau2, sc2;
      long long beta;
      fx_reflect(alpha.x, alpha.y, n2, 104 + 2 * M, ev, tau2, sc2, beta);
      if (lane == 0) {   // v = x sc = 2 (x 2^ev) (sc 2^-ev / 2)
        s_sc = sc2;
        s_ev = ev;
        s_beta[jn] = beta;
        s_bev[jn] = -ev;
        s_tau[jn] = tau2;
      }
      if (lane > jn && lane < jb) {
        // -conj(tau) (row_k + conj(sc) S_k) = -4 conj(tau/2) (row_k/2 + conj(sc 2^-ev/2) (S_k 2^ev))
        auto scaled = [&](long long S) { return ev >= M ? S << (ev - M) : fx_shr(S, M - ev); };
        const longlong2 row = s_rowin[par][lane];
        longlong2 w = make_longlong2((row.x + 1) >> 1, (row.y + 1) >> 1);
        w = fx_cfma(w, fx(sc2.x), fx(-sc2.y), fx(sc2.y), fx(scaled(Sk.x)), fx(scaled(Sk.y)));
        const longlong2 f = fx_cfma(make_longlong2(0, 0), fx(tau2.x), fx(-tau2.y), fx(tau2.y), fx(w.x), fx(w.y));
        const Fx gr = fw(-(f.x << 4)), gi = fw(-(f.y << 4)), gn = fw(f.y << 4);   // f 4, and the products' 2^2
        s_g[lane] = make_int4(gr.h, gr.l, gi.h, gi.l);
        s_gn[lane] = make_int2(gn.h, gn.l);
      }
    }
    __syncthreads();
  }
  // back to doubles: v below the diagonal, the scaled R above it
  for (int r = rbeg + lane % RW, x = xbeg; r < W; r += rstep, x += xstep)
#pragma unroll
    for (int k = 0; k < HB; ++k) {
      const int col = Q * k + q;
      if (col >= jb) continue;
      const longlong2 a = Zx[x + (size_t)col * ldx];
      const int e2 = r > j0 + col ? 0 : s_exp[col];
      double2 z = make_double2(fx_to(a.x, e2), fx_to(a.y, e2));
      if (r == j0 + col) z = make_double2(fx_to(s_beta[col], s_exp[col] + s_bev[col]), 0.0);
      if (col >= s_bad) z = make_double2(nan(""), nan(""));
      p.Z[r + (size_t)(j0 + col) * ld] = z;
    }
  if (rank == 0 && tid < jb)
    p.T[tid] = make_double2(tid < s_bad ? fx_to(s_tau[tid].x, 1) : nan(""), tid < s_bad ? fx_to(s_tau[tid].y, 1) : 0.0);
  cluster.sync();   // no CTA leaves while another may still read its partial sums
}

// Trailing update Q^H C = C - V (T^H (V^H C)) for every 32-column tile of
// the trailing block, in three launches so that the rows of a tall matrix
// spread over many CTAs: partial products Y_b = V_b^H C_b of each block of
// QR_RB rows; their sum (fixed order) times T^H; C_b -= V_b Y.
template <typename C>
__global__ void __launch_bounds__(UT) k_qr_ypart(const QrProb<C>* __restrict__ P, int j0) {
  const QrProb<C> p = P[blockIdx.z];
  if (j0 >= p.n) return;
  const int jb = min(QR_NB, p.n - j0);
  const int tile = blockIdx.x, rb = blockIdx.y;
  const int c0 = j0 + jb + tile * 32;
  const int rbeg = j0 + rb * QR_RB;
  if (c0 >= p.n || rbeg >= p.W) return;
  const int nc = min(32, p.n - c0), rend = min(p.W, rbeg + QR_RB);
  const int tid = threadIdx.x;
  __shared__ C s_v[RC][QR_NB + 1];
  __shared__ C s_c[RC][33];
  const int tx = tid & 15, ty = tid >> 4;
  C y00 = czero<C>(), y01 = czero<C>(), y10 = czero<C>(), y11 = czero<C>();
  for (int r0 = rbeg; r0 < rend; r0 += RC) {
    for (int e = tid; e < RC * 32; e += UT) {
      const int i = e % RC, j = e / RC, r = r0 + i;
      s_v[i][j] = r < rend ? v_entry(p, j0, jb, r, j) : czero<C>();
      s_c[i][j] = (j < nc && r < rend) ? p.Z[r + (size_t)(c0 + j) * p.ld] : czero<C>();
    }
    __syncthreads();
#pragma unroll 8
    for (int i = 0; i < RC; ++i) {
      const C a0 = s_v[i][tx], a1 = s_v[i][tx + 16], b0 = s_c[i][ty], b1 = s_c[i][ty + 16];
      cfma_conj(y00, a0, b0); cfma_conj(y01, a0, b1);
      cfma_conj(y10, a1, b0); cfma_conj(y11, a1, b1);
    }
    __syncthreads();
  }
  C* yp = p.Yp + ((size_t)tile * p.mrb + rb) * (QR_NB * 32);
  yp[tx + QR_NB * ty] = y00;
  yp[tx + QR_NB * (ty + 16)] = y01;
  yp[tx + 16 + QR_NB * ty] = y10;
  yp[tx + 16 + QR_NB * (ty + 16)] = y11;
}

// Y = sum of the row blocks' partials (in block order), then T^H Y into the
// tile's first partial slot.
template <typename C>
__global__ void __launch_bounds__(UT) k_qr_yreduce(const QrProb<C>* __restrict__ P, int j0) {
  const QrProb<C> p = P[blockIdx.y];
  if (j0 >= p.n) return;
  const int jb = min(QR_NB, p.n - j0);
  const int tile = blockIdx.x;
  if (j0 + jb + tile * 32 >= p.n) return;
  const int nrb = (p.W - j0 + QR_RB - 1) / QR_RB;
  const int tid = threadIdx.x;
  __shared__ C s_y[QR_NB][33];
  __shared__ C s_t[QR_NB][QR_NB + 1];
  C* yp = p.Yp + (size_t)tile * p.mrb * (QR_NB * 32);
  for (int e = tid; e < QR_NB * 32; e += UT) {
    C acc = czero<C>();
    for (int b = 0; b < nrb; ++b) acc = acc + yp[(size_t)b * (QR_NB * 32) + e];
    s_y[e % QR_NB][e / QR_NB] = acc;
  }
  for (int e = tid; e < QR_NB * QR_NB; e += UT) s_t[e % QR_NB][e / QR_NB] = p.T[e];
  __syncthreads();
  for (int e = tid; e < QR_NB * 32; e += UT) {
    const int i = e % QR_NB, cc = e / QR_NB;
    C acc = czero<C>();
    for (int l = 0; l <= i; ++l) cfma_conj(acc, s_t[l][i], s_y[l][cc]);
    yp[e] = acc;
  }
}

template <typename C>
__global__ void __launch_bounds__(UT) k_qr_apply(const QrProb<C>* __restrict__ P, int j0) {
  const QrProb<C> p = P[blockIdx.z];
  if (j0 >= p.n) return;
  const int jb = min(QR_NB, p.n - j0);
  const int tile = blockIdx.x, rb = blockIdx.y;
  const int c0 = j0 + jb + tile * 32;
  const int rbeg = j0 + rb * QR_RB;
  if (c0 >= p.n || rbeg >= p.W) return;
  const int nc = min(32, p.n - c0), rend = min(p.W, rbeg + QR_RB);
  const int tid = threadIdx.x;
  __shared__ C s_v[RC][QR_NB + 1];
  __shared__ C s_y[QR_NB][33];
  const C* yp = p.Yp + (size_t)tile * p.mrb * (QR_NB * 32);
  for (int e = tid; e < QR_NB * 32; e += UT) s_y[e % QR_NB][e / QR_NB] = yp[e];
  const int ri = tid & 31, g = tid >> 5;
  for (int r0 = rbeg; r0 < rend; r0 += RC) {
    __syncthreads();
    for (int e = tid; e < RC * QR_NB; e += UT) {
      const int i = e % RC, j = e / RC;
      s_v[i][j] = v_entry(p, j0, jb, r0 + i, j);
    }
    __syncthreads();
    C acc[4] = {czero<C>(), czero<C>(), czero<C>(), czero<C>()};
    for (int j = 0; j < jb; ++j) {
      const C v = s_v[ri][j];
#pragma unroll
      for (int q = 0; q < 4; ++q) cfma(acc[q], v, s_y[j][4 * g + q]);
    }
    const int r = r0 + ri;
    if (r < rend) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (4 * g + q < nc) {
          C* pz = p.Z + r + (size_t)(c0 + 4 * g + q) * p.ld;
          *pz = *pz - acc[q];
        }
    }
  }
}

// C_b -= V_b Y on the fifth-generation tensor cores (complex64, the default
// path): one CTA per 64-row block of a matrix walks all 32-column tiles of
// its trailing block.  The complex product is a real one of twice the size,
// [Re D; Im D] = [[Re V, -Im V], [Im V, Re V]] [Re Y; Im Y], i.e. an
// M = 128, N = 32, K = 64 real MMA; every FP32 operand is split into tf32
// parts x = hi + lo and hi*hi + hi*lo + lo*hi are accumulated in FP32 (the
// 3xTF32 scheme, FP32 accuracy), and each tile's accumulation is only 64
// real terms long.  V_b is split into shared memory once; per tile the CTA
// stages Y (from the row-block reduction) into one of two buffers, one
// thread issues the 24 MMAs into one of two TMEM accumulators and commits
// them to that buffer's mbarrier, and the epilogue of the previous tile
// (tcgen05.ld by all eight warps, each with a quarter of the rows and half
// of the columns, then each thread's component of C -= D, with C loaded one
// tile ahead) overlaps them.  Every wait is bounded; a wait that runs out
// sets *err and the CTA stops writing.
namespace tcq {
constexpr int T = 256;                         // threads: warp w reads TMEM lanes [32 (w % 4), + 32), columns 16 (w / 4) ..
constexpr int ROWS = 64;                       // complex rows per CTA
constexpr int KR = 2 * QR_NB;                  // real k: real and imaginary parts of the reflectors
constexpr uint32_t A_BYTES = 2 * ROWS * KR * 4;    // one of hi / lo: 128 x 64 tf32
constexpr uint32_t B_BYTES = 32 * KR * 4;          // one of hi / lo: 32 x 64 tf32
constexpr uint32_t OFF_B = 2 * A_BYTES;            // two buffers of (hi, lo)
constexpr uint32_t OFF_BAR = OFF_B + 4 * B_BYTES;
constexpr int SMEM = OFF_BAR + 64;
constexpr uint32_t IDESC = tcx::idesc_tf32(2 * ROWS, 32);
constexpr uint32_t TMEM_COLS = 64;             // two 32-column accumulators
constexpr int WAIT = 1 << 20;                  // x ~1 us suspend hint: about a second
}  // namespace tcq

// no_arrive (tests of the timeout path): every CTA first waits, with a bound
// of about a millisecond, on a barrier that nothing arrives at, then issues
// nothing, frees its tensor memory and sets *err.
// At most 112 registers: two CTAs per SM beside one CTA of the operator assembly.
__global__ void __maxnreg__(112) k_qr_apply_tc(const QrProb<float2>* __restrict__ P, int j0, int* err,
                                                        int no_arrive) {
  using namespace tcq;
  extern __shared__ __align__(1024) unsigned char sm[];
  const QrProb<float2> p = P[blockIdx.y];
  if (j0 >= p.n) return;
  const int jb = min(QR_NB, p.n - j0);
  const int cfirst = j0 + jb;
  const int ntiles = (p.n - cfirst + 31) / 32;
  const int rbeg = j0 + (int)blockIdx.x * ROWS;
  if (ntiles <= 0 || rbeg >= p.W) return;
  const int rend = min(p.W, rbeg + ROWS);
  const int tid = threadIdx.x, warp = tid >> 5;
  unsigned char* Ahi = sm;
  unsigned char* Alo = sm + A_BYTES;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + OFF_BAR);
  uint32_t* s_taddr = reinterpret_cast<uint32_t*>(sm + OFF_BAR + 24);
  if (tid == 0) {
    tcx::mbar_init(&mbar[0]);
    tcx::mbar_init(&mbar[1]);
    tcx::mbar_init(&mbar[2]);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tcx::smem_u32(s_taddr)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // A: the block's reflector rows (unit diagonal, zeros above it and past W)
#pragma unroll 4
  for (int i = 0; i < 8; ++i) {
    const int mm = tid & 63, kk = (tid >> 6) + 4 * i;
    const float2 v = v_entry(p, j0, jb, rbeg + mm, kk);
    tcx::put_split(Ahi, Alo, tcx::core_off<KR>(mm, kk), v.x);
    tcx::put_split(Ahi, Alo, tcx::core_off<KR>(mm, QR_NB + kk), -v.y);
    tcx::put_split(Ahi, Alo, tcx::core_off<KR>(ROWS + mm, kk), v.y);
    tcx::put_split(Ahi, Alo, tcx::core_off<KR>(ROWS + mm, QR_NB + kk), v.x);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *s_taddr;
  bool ok = true;
  if (no_arrive) ok = tcx::mbar_wait(&mbar[2], 0, 1 << 10);
  const int nt = __syncthreads_and(ok ? 1 : 0) ? ntiles : -1;
  // Epilogue work split: warp w reads TMEM lanes 32 (w % 4) .. + 32, i.e.
  // D's real row lane = 32 (w % 4) + (tid & 31): the real (lane < 64) or
  // imaginary (lane >= 64) part of complex row rbeg + (lane & 63), columns
  // 16 (w / 4) .. + 16 of the tile; each thread updates that component of C
  // itself (no exchange).  C of tile t is loaded at iteration t and updated
  // at iteration t + 1, and Y of tile t + 1 is loaded at iteration t, so
  // their latency overlaps the MMAs and the previous epilogue.
  const int lane_row = 32 * (warp & 3) + (tid & 31), hcol = 16 * (warp >> 2);
  const int r = lane_row & 63, comp = lane_row >> 6;
  const int row = rbeg + r;
  const bool row_ok = row < rend;
  float cnext[16], ccur[16];
  float2 ynext[4];
  auto load_y = [&](int t) {
    const float2* yp = p.Yp + (size_t)t * p.mrb * (QR_NB * 32);
#pragma unroll
    for (int i = 0; i < 4; ++i) ynext[i] = yp[(tid & 31) + QR_NB * ((tid >> 5) + 8 * i)];
  };
  if (nt > 0) load_y(0);
  for (int t = 0; t <= nt; ++t) {
    if (t < nt) {
      const int b = t & 1;
      unsigned char* Bhi = sm + OFF_B + b * 2 * B_BYTES;
      unsigned char* Blo = Bhi + B_BYTES;
      // Y of tile t (rows: reflectors, columns: the tile's columns), stored transposed;
      // buffer b was last read by the MMAs of tile t - 2, waited for at iteration t - 1
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int kk = tid & 31, nn = (tid >> 5) + 8 * i;
        tcx::put_split(Bhi, Blo, tcx::core_off<KR>(nn, kk), ynext[i].x);
        tcx::put_split(Bhi, Blo, tcx::core_off<KR>(nn, QR_NB + kk), ynext[i].y);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncthreads();
      if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t acc = tmem + (uint32_t)(b * 32);
        const uint32_t ah = tcx::smem_u32(Ahi), al = tcx::smem_u32(Alo);
        const uint32_t bh = tcx::smem_u32(Bhi), bl = tcx::smem_u32(Blo);
#pragma unroll
        for (int s = 0; s < KR / 8; ++s) {
          const uint32_t o = s * 2 * tcx::LBO;   // 8 tf32 along k = two core matrices
          tcx::mma_tf32<IDESC>(acc, tcx::sdesc<KR>(ah + o), tcx::sdesc<KR>(bh + o), s > 0 ? 1u : 0u);
          tcx::mma_tf32<IDESC>(acc, tcx::sdesc<KR>(ah + o), tcx::sdesc<KR>(bl + o), 1u);
          tcx::mma_tf32<IDESC>(acc, tcx::sdesc<KR>(al + o), tcx::sdesc<KR>(bh + o), 1u);
        }
        tcx::mma_commit(&mbar[b]);
      }
      if (t + 1 < nt) load_y(t + 1);
      // this thread's component of C, tile t, its 16 columns
      const int c0 = cfirst + t * 32 + hcol, nc = min(16, p.n - c0);
      const float* cz = reinterpret_cast<const float*>(p.Z + row + (size_t)c0 * p.ld) + comp;
#pragma unroll
      for (int j = 0; j < 16; ++j) cnext[j] = (row_ok && j < nc) ? cz[(size_t)j * 2 * p.ld] : 0.f;
    }
    if (t >= 1) {   // epilogue of tile u = t - 1
      const int u = t - 1, b = u & 1;
      ok = ok && tcx::mbar_wait(&mbar[b], (uint32_t)((u >> 1) & 1), WAIT);   // after a failure: no more waits
      asm volatile("tcgen05.fence::after_thread_sync;");
      float d[16];
      const bool wok = __all_sync(0xffffffffu, ok ? 1 : 0);
      if (wok) {
        tcx::tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * 32 + hcol), d);
        const int c0 = cfirst + u * 32 + hcol, nc = min(16, p.n - c0);
        float* cz = reinterpret_cast<float*>(p.Z + row + (size_t)c0 * p.ld) + comp;
        if (row_ok) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (j < nc) cz[(size_t)j * 2 * p.ld] = ccur[j] - d[j];
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) ccur[j] = cnext[j];
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  const int all_ok = __syncthreads_and(ok ? 1 : 0);
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  if (!all_ok && tid == 0) atomicExch(err, 1);
}

// ---- complex128 trailing update on the tensor cores (oz.cuh) -----------------------
// Y^H = [V | C]^H V in partial sums over blocks of OZ_RB rows (one CTA per 128
// columns from j0 on and row block), their sum with T^H applied, C -= V Y.

// Partial (columns i, reflectors j): sum over the block's rows of conj(X_i) V_j, X the panel's V, then C.
__global__ void __launch_bounds__(oz::T) k_qr_oz_ypart(const QrProb<double2>* __restrict__ P, int j0, int* err,
                                                       int no_arrive) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const QrProb<double2> p = P[blockIdx.z];
  const int c0 = j0 + (int)blockIdx.x * oz::TM, rbeg = j0 + (int)blockIdx.y * OZ_RB;
  if (j0 + QR_NB >= p.n || c0 >= p.n || rbeg >= p.W) return;   // no trailing columns: no update
  const int rend = min(p.W, rbeg + OZ_RB);
  double2 acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = czero<double2>();
  oz::Cta cta = oz::begin(sm, no_arrive);
  for (int r0 = rbeg; r0 < rend; r0 += oz::TKC)
    oz::stage(cta, true,
                    [&](int i, int l) {
                      const int c = c0 + i, r = r0 + l;
                      if (c >= p.n || r >= rend) return czero<double2>();
                      return conj(c < j0 + QR_NB ? v_entry(p, j0, QR_NB, r, c - j0) : p.Z[r + (size_t)c * p.ld]);
                    },
                    [&](int l, int j) { return r0 + l < rend ? v_entry(p, j0, QR_NB, r0 + l, j) : czero<double2>(); },
                    [&](int j, int part, double d) { if (part == 0) acc[j].x += d; else acc[j].y += d; }, [] {});
  const int warp = threadIdx.x >> 5, i = 32 * (warp & 3) + (threadIdx.x & 31), cgp = 8 * (warp >> 2);
  double2* yp = p.Yp + ((size_t)blockIdx.x * p.mrb + blockIdx.y) * (oz::TM * QR_NB);
  if (cta.ok) {
#pragma unroll
    for (int j = 0; j < 8; ++j) yp[i + oz::TM * (cgp + j)] = acc[j];
  }
  oz::end(cta, err);
}

// Y = T^H (V^H C) for 32 columns: the partials summed in row-block order, then
// T^{-H} x = y solved forward (T^{-1} = diag(1/tau) + the strict upper part of
// V^H V), a warp per column and a lane per reflector.
__global__ void __launch_bounds__(UT) k_qr_oz_yreduce(const QrProb<double2>* __restrict__ P, int j0) {
  const QrProb<double2> p = P[blockIdx.y];
  const int cbeg = QR_NB + 32 * (int)blockIdx.x;   // column offset from j0
  if (j0 + cbeg >= p.n) return;
  const int nrb = (p.W - j0 + OZ_RB - 1) / OZ_RB;
  __shared__ double2 s_g[QR_NB][QR_NB + 1];        // G[l][j] = v_l^H v_j
  const int tid = threadIdx.x, lane = tid & 31;
  for (int e = tid; e < QR_NB * QR_NB; e += UT) {
    const int l = e % QR_NB, j = e / QR_NB;
    double2 a = czero<double2>();
    if (l < j)
      for (int b = 0; b < nrb; ++b) a = a + p.Yp[(size_t)b * (oz::TM * QR_NB) + l + oz::TM * j];
    s_g[l][j] = a;
  }
  const double2 ctau = conj(p.T[lane]);
  __syncthreads();
  for (int w = tid >> 5; w < 32; w += UT / 32) {
    const int o = cbeg + w;
    if (j0 + o >= p.n) continue;
    const double2* yp = p.Yp + (size_t)(o / oz::TM) * p.mrb * (oz::TM * QR_NB) + o % oz::TM + oz::TM * lane;
    double2 x = czero<double2>();
    for (int b = 0; b < nrb; ++b) x = x + yp[(size_t)b * (oz::TM * QR_NB)];
    x = conj(x);
    for (int l = 0; l < QR_NB; ++l) {
      if (lane == l) x = ctau * x;
      const double2 xl = make_double2(__shfl_sync(0xffffffffu, x.x, l), __shfl_sync(0xffffffffu, x.y, l));
      if (lane > l) {
        const double2 g = s_g[l][lane];
        x.x = fma(-g.x, xl.x, x.x); x.x = fma(-g.y, xl.y, x.x);   // x -= conj(g) xl
        x.y = fma(-g.x, xl.y, x.y); x.y = fma(g.y, xl.x, x.y);
      }
    }
    p.V[lane + (size_t)QR_NB * (o - QR_NB)] = x;   // Y, QR_NB x trailing columns
  }
}

__global__ void __launch_bounds__(oz::T) k_qr_oz_apply(const QrProb<double2>* __restrict__ P, int j0, int per, int* err,
                                                       int no_arrive) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const QrProb<double2> p = P[blockIdx.z];
  const int cfirst = j0 + QR_NB, r0 = j0 + (int)blockIdx.x * oz::TM, t0 = (int)blockIdx.y * per;
  if (cfirst + t0 * oz::TN >= p.n || r0 >= p.W) return;
  const int t1 = min(t0 + per, (p.n - cfirst + oz::TN - 1) / oz::TN);
  const int warp = threadIdx.x >> 5, row = r0 + 32 * (warp & 3) + (threadIdx.x & 31), cgp = 8 * (warp >> 2);
  oz::Cta cta = oz::begin(sm, no_arrive);
  for (int t = t0; t < t1; ++t) {
    const int c0 = t * oz::TN;   // trailing column
    double2 z[8];   // C, minus the products
    oz::stage(cta, t == t0, [&](int i, int l) { return v_entry(p, j0, QR_NB, r0 + i, l); },
                     [&](int l, int j) {
                       return cfirst + c0 + j < p.n ? p.V[l + (size_t)QR_NB * (c0 + j)] : czero<double2>();
                     },
                     [&](int j, int part, double d) { if (part == 0) z[j].x -= d; else z[j].y -= d; },
                     [&] {
#pragma unroll
                       for (int j = 0; j < 8; ++j)
                         z[j] = row < p.W && cfirst + c0 + cgp + j < p.n ? p.Z[row + (size_t)(cfirst + c0 + cgp + j) * p.ld]
                                                                         : czero<double2>();
                     });
    if (row < p.W && cta.ok) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (cfirst + c0 + cgp + j < p.n) p.Z[row + (size_t)(cfirst + c0 + cgp + j) * p.ld] = z[j];
    }
  }
  oz::end(cta, err);
}

// Zeros below the diagonal of the top n x n block (the reflectors' storage).
template <typename C>
__global__ void k_qr_zero_lower(const QrProb<C>* __restrict__ P) {
  const QrProb<C> p = P[blockIdx.y];
  const int j = blockIdx.x;
  if (j >= p.n) return;
  C* col = p.Z + (size_t)j * p.ld;
  for (int r = j + 1 + threadIdx.x; r < p.n; r += blockDim.x) col[r] = czero<C>();
}

}  // namespace

template <typename C>
void qr_panel(const QrProb<C>* d_prob, int nprob, int j0, cudaStream_t st, int cluster, int max_w) {
  if (nprob <= 0) return;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // cluster of up to 8 CTAs per matrix, enough to fill the SMs (one CTA per SM)
  int cs = 1;
  if (cluster > 0) cs = cluster;
  else
    while (cs < 8 && (long)nprob * cs * 2 <= sms) cs *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nprob * cs);
  cfg.blockDim = dim3(PT);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  KPROF_BEGIN(st);
  if constexpr (std::is_same<C, double2>::value) {
    const int sweeps = (max_w - j0 + PanelSplit<4>::PR * cs - 1) / (PanelSplit<4>::PR * cs), ldp = sweeps * PanelSplit<4>::PR;
    if (sweeps <= FX_SWEEPS) {
      cfg.dynamicSmemBytes = (size_t)ldp * QR_NB * sizeof(double2);
      // the same value every time: idempotent across threads and devices
      cudaFuncSetAttribute(k_qr_panel_fx<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(FX_SWEEPS * PanelSplit<4>::PR * QR_NB * sizeof(double2)));
      cudaLaunchKernelEx(&cfg, k_qr_panel_fx<true>, d_prob, j0, ldp);
    } else {
      cudaLaunchKernelEx(&cfg, k_qr_panel_fx<false>, d_prob, j0, 0);
    }
  } else {
    auto rows = [&](int c) { return ((max_w - j0 + c - 1) / c + 31) & ~31; };
    while (cs < 8 && rows(cs) > SUB_ROWS) cs *= 2;   // the sub-panels in shared memory
    cfg.gridDim = dim3(nprob * cs);
    attr[0].val.clusterDim.x = cs;
    if (max_w > 0 && rows(cs) <= SUB_ROWS) {
      cfg.dynamicSmemBytes = PANEL_RED + (size_t)rows(cs) * SB * sizeof(C);
      // the same value every time: idempotent across threads and devices
      cudaFuncSetAttribute(k_qr_panel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(PANEL_RED + (size_t)SUB_ROWS * SB * sizeof(C)));
      cudaLaunchKernelEx(&cfg, k_qr_panel<true>, d_prob, j0, rows(cs));
    } else {
      cfg.dynamicSmemBytes = PANEL_RED;
      cudaFuncSetAttribute(k_qr_panel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PANEL_RED);
      cudaLaunchKernelEx(&cfg, k_qr_panel<false>, d_prob, j0, 0);
    }
  }
  pm_launch_count_add(1);
  KPROF_END(st, kname<C>("qr_panel", "qr_panel32"), 0.0);
}
template <typename C>
void qr_update(const QrProb<C>* d_prob, int nprob, int j0, int max_tiles, int max_rb, cudaStream_t st,
               int* tc_err, int max_w, bool no_arrive) {
  if (nprob <= 0 || max_tiles <= 0 || max_rb <= 0) return;
  KPROF_BEGIN(st);
  k_qr_ypart<C><<<dim3(max_tiles, max_rb, nprob), UT, 0, st>>>(d_prob, j0);
  k_qr_yreduce<C><<<dim3(max_tiles, nprob), UT, 0, st>>>(d_prob, j0);
  bool on_tc = false;
  if constexpr (std::is_same<C, float2>::value) {
    if (tc_err) {
      // the same value every time: idempotent across threads and devices
      cudaFuncSetAttribute(k_qr_apply_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, tcq::SMEM);
      const int rblocks = (max_w - j0 + tcq::ROWS - 1) / tcq::ROWS;
      if (rblocks > 0) k_qr_apply_tc<<<dim3(rblocks, nprob), tcq::T, tcq::SMEM, st>>>(d_prob, j0, tc_err,
                                                                                       no_arrive ? 1 : 0);
      on_tc = true;
    }
  }
  if (!on_tc) k_qr_apply<C><<<dim3(max_tiles, max_rb, nprob), UT, 0, st>>>(d_prob, j0);
  pm_launch_count_add(3);
  KPROF_END(st, on_tc ? "qr_update_tc32" : kname<C>("qr_update", "qr_update32"), 0.0);
}
void qr_update_oz(const QrProb<double2>* d_prob, int nprob, int j0, int max_n, int max_w, int* err, cudaStream_t st) {
  const int nt = max_n - j0 - QR_NB;
  if (nprob <= 0 || nt <= 0) return;
  // the same value every time: idempotent across threads and devices
  cudaFuncSetAttribute(k_qr_oz_ypart, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM);
  cudaFuncSetAttribute(k_qr_oz_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM);
  const int rbs = (max_w - j0 + OZ_RB - 1) / OZ_RB, mt = (max_w - j0 + oz::TM - 1) / oz::TM;
  const int tiles = (nt + oz::TN - 1) / oz::TN, per = oz_per((long)mt * tiles * nprob);
  KPROF_BEGIN(st);
  k_qr_oz_ypart<<<dim3((max_n - j0 + oz::TM - 1) / oz::TM, rbs, nprob), oz::T, oz::SMEM, st>>>(d_prob, j0, err,
                                                                                                   g_oz_no_arrive);
  k_qr_oz_yreduce<<<dim3(tiles, nprob), UT, 0, st>>>(d_prob, j0);
  k_qr_oz_apply<<<dim3(mt, (tiles + per - 1) / per, nprob), oz::T, oz::SMEM, st>>>(d_prob, j0, per, err,
                                                                                    g_oz_no_arrive);
  pm_launch_count_add(3);
  KPROF_END(st, "qr_update_oz", 0.0);
}
template <typename C>
void qr_zero_lower(const QrProb<C>* d_prob, int nprob, int max_n, cudaStream_t st) {
  if (nprob <= 0 || max_n <= 0) return;
  k_qr_zero_lower<C><<<dim3(max_n, nprob), 256, 0, st>>>(d_prob);
  pm_launch_count_add(1);
}

template void qr_panel<float2>(const QrProb<float2>*, int, int, cudaStream_t, int, int);
template void qr_panel<double2>(const QrProb<double2>*, int, int, cudaStream_t, int, int);
template void qr_zero_lower<double2>(const QrProb<double2>*, int, int, cudaStream_t);
template void qr_update<float2>(const QrProb<float2>*, int, int, int, int, cudaStream_t, int*, int, bool);
template void qr_zero_lower<float2>(const QrProb<float2>*, int, int, cudaStream_t);
