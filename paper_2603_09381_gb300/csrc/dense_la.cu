// Batched complex GEMM / LU / LU-solve kernels.
//
// complex128 products and trailing updates run on the tensor cores (oz_gemm.cuh);
// what is left to the FP64 pipe here (about 1.2 TFLOP/s: even a rank-1 update
// streamed from HBM is bound by it) are panels, diagonal blocks, chained solves
// and products of a few rows, columns or terms.  complex64 updates and products
// run on the FP32 pipe, in shared-memory tiles.
#include "dense_la.cuh"
#include "oz_gemm.cuh"
#include "prof.cuh"
#include <type_traits>
#include <algorithm>
#include <vector>
#include <cooperative_groups.h>

namespace {

constexpr int TB = 32;   // output tile
constexpr int TK = 16;   // k step
constexpr int MAXNB = 32;   // panel width of the LU kernels

// One 32 x 32 output tile of  Cm = alpha * A * B + beta * Cm  (256 threads).
// SUB: the caller's alpha = -1 and beta = 1, applied as Cm - A * B (the same
// bits: multiplying by (-1, 0) and (1, 0) is exact), which spares the
// epilogue's complex multiplications (an eighth of an update's FP64 work at
// k = 16).
template <typename C, bool SUB = false>
__device__ __forceinline__ void gemm_tile(int m, int n, int k, const C* __restrict__ A, int lda,
                                          const C* __restrict__ B, int ldb, C* Cm, int ldc,
                                          C alpha, C beta, int beta_zero, int tm, int tn) {
  __shared__ C As[TK][TB + 1];
  __shared__ C Bs[TK][TB + 1];
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int r0 = tm * TB, c0 = tn * TB;
  C acc00 = czero<C>(), acc01 = czero<C>(), acc10 = czero<C>(), acc11 = czero<C>();
  for (int l0 = 0; l0 < k; l0 += TK) {
    for (int e = tid; e < TB * TK; e += 256) {
      int i = e % TB, l = e / TB;
      int gi = r0 + i, gl = l0 + l;
      As[l][i] = (gi < m && gl < k) ? A[gi + (size_t)gl * lda] : czero<C>();
    }
    for (int e = tid; e < TB * TK; e += 256) {
      int l = e % TK, j = e / TK;
      int gl = l0 + l, gj = c0 + j;
      Bs[l][j] = (gl < k && gj < n) ? B[gl + (size_t)gj * ldb] : czero<C>();
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < TK; ++l) {
      C a0 = As[l][tx], a1 = As[l][tx + 16];
      C b0 = Bs[l][ty], b1 = Bs[l][ty + 16];
      cfma(acc00, a0, b0); cfma(acc01, a0, b1);
      cfma(acc10, a1, b0); cfma(acc11, a1, b1);
    }
    __syncthreads();
  }
  C accs[2][2] = {{acc00, acc01}, {acc10, acc11}};
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      int gi = r0 + tx + 16 * a, gj = c0 + ty + 16 * b;
      if (gi < m && gj < n) {
        C* p = Cm + gi + (size_t)gj * ldc;
        if (SUB) {
          *p = *p - accs[a][b];
        } else {
          C v = alpha * accs[a][b];
          if (!beta_zero) v = v + beta * (*p);
          *p = v;
        }
      }
    }
}

template <typename C>
__global__ void __launch_bounds__(256) k_gemm_batched(const GemmDesc<C>* __restrict__ d,
                                                      const int* __restrict__ tile_off, int nprob) {
  int t = blockIdx.x;
  int lo = 0, hi = nprob;  // find prob with tile_off[prob] <= t < tile_off[prob+1]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (tile_off[mid] <= t) lo = mid; else hi = mid;
  }
  const GemmDesc<C> g = d[lo];
  int local = t - tile_off[lo];
  int tiles_m = (g.m + TB - 1) / TB;
  if (g.m <= 0 || g.n <= 0) return;
  gemm_tile<C>(g.m, g.n, g.k, g.A, g.lda, g.B, g.ldb, g.Cm, g.ldc, g.alpha, g.beta, g.beta_zero,
               local % tiles_m, local / tiles_m);
}

// The same product with a TM x TN output tile, each of the 256 threads
// holding MR x NR outputs (TM / MR by TN / NR threads).  Every output
// accumulates over k in the same order as gemm_tile (chunks of TK, each in
// order), so all tile shapes give bit-identical results; the autotuner picks
// among them by speed alone.
template <typename C, int TM, int TN, int MR, int NR>
__device__ __forceinline__ void gemm_tile_t(int m, int n, int k, const C* __restrict__ A, int lda,
                                            const C* __restrict__ B, int ldb, C* Cm, int ldc, C alpha, C beta,
                                            int beta_zero, int r0, int c0) {
  constexpr int TX = TM / MR, TY = TN / NR;
  static_assert(TX * TY == 256, "256 threads per tile");
  __shared__ C As[TK][TM + 1];
  __shared__ C Bs[TK][TN + 1];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  C acc[MR][NR];
#pragma unroll
  for (int a = 0; a < MR; ++a)
#pragma unroll
    for (int b = 0; b < NR; ++b) acc[a][b] = czero<C>();
  for (int l0 = 0; l0 < k; l0 += TK) {
    for (int e = tid; e < TM * TK; e += 256) {
      const int i = e % TM, l = e / TM;
      const int gi = r0 + i, gl = l0 + l;
      As[l][i] = (gi < m && gl < k) ? A[gi + (size_t)gl * lda] : czero<C>();
    }
    for (int e = tid; e < TN * TK; e += 256) {
      const int l = e % TK, j = e / TK;
      const int gl = l0 + l, gj = c0 + j;
      Bs[l][j] = (gl < k && gj < n) ? B[gl + (size_t)gj * ldb] : czero<C>();
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < TK; ++l) {
      C av[MR], bv[NR];
#pragma unroll
      for (int a = 0; a < MR; ++a) av[a] = As[l][tx + TX * a];
#pragma unroll
      for (int b = 0; b < NR; ++b) bv[b] = Bs[l][ty + TY * b];
#pragma unroll
      for (int a = 0; a < MR; ++a)
#pragma unroll
        for (int b = 0; b < NR; ++b) cfma(acc[a][b], av[a], bv[b]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < MR; ++a)
#pragma unroll
    for (int b = 0; b < NR; ++b) {
      const int gi = r0 + tx + TX * a, gj = c0 + ty + TY * b;
      if (gi < m && gj < n) {
        C* p = Cm + gi + (size_t)gj * ldc;
        C v = alpha * acc[a][b];
        if (!beta_zero) v = v + beta * (*p);
        *p = v;
      }
    }
}

template <typename C, int TM, int TN, int MR, int NR>
__global__ void __launch_bounds__(256) k_gemm_batched_t(const GemmDesc<C>* __restrict__ d,
                                                        const int* __restrict__ tile_off, int nprob) {
  const int t = blockIdx.x;
  int lo = 0, hi = nprob;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tile_off[mid] <= t) lo = mid; else hi = mid;
  }
  const GemmDesc<C> g = d[lo];
  if (g.m <= 0 || g.n <= 0) return;
  const int local = t - tile_off[lo];
  const int tiles_m = (g.m + TM - 1) / TM;
  gemm_tile_t<C, TM, TN, MR, NR>(g.m, g.n, g.k, g.A, g.lda, g.B, g.ldb, g.Cm, g.ldc, g.alpha, g.beta, g.beta_zero,
                                 (local % tiles_m) * TM, (local / tiles_m) * TN);
}

// ---- LU with partial pivoting (blocked, right-looking) ---------------------------------

__device__ __forceinline__ double2 shfl_c(double2 v, int src) {
  return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ float2 shfl_c(float2 v, int src) {
  return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// Panel: columns [p, p + jb) of rows [p, m) on a cluster of CTAs per matrix,
// right-looking.  One FP64 pipe does 2 fused multiply-adds per clock, so a
// panel on one SM is bound by it however small the matrix (512 rows: 15 us a
// column); over 8 SMs the update of a column shrinks to the cost of its
// barriers.  The rows go to the CTAs in cyclic chunks of 32 and stay there, in
// shared memory when they fit (SM), else in place.  Per column: every CTA
// writes its largest |a|^2 (lowest row on ties) and a copy of that row to every
// CTA's shared memory, rank 0, which owns the diagonal rows, a copy of the
// diagonal row; one cluster barrier; every CTA takes the winner's row as the
// row of U, the two owners swap, and a -= (a_jj / pivot) u on each CTA's rows.
// The column itself is divided by its pivot when the panel is written back.
// An entry's operations do not depend on the number of CTAs, so neither do the
// bits.  The comparisons run on the integer pipe (non-negative floats
// order like their bit patterns).
// complex64: a step updates its group of 8 columns only.  At a group's end the
// columns to its right take the group's eight products as one sum (every CTA has
// kept the pivot rows and solves for the rows of U itself), so that an entry is
// rounded once a group and not at every column: the backward error of a system of 80 to 400
// unknowns is 0.9e-7, as with the sums of 16 columns that came before, against
// 1.5e-7 column by column.  complex128 goes column by column: its updates outside
// the panel are rounded once for 32 columns.
constexpr int LP_T = 256;
template <typename R> constexpr int LP_GROUP = sizeof(R) == 4 ? 8 : MAXNB;
template <typename C, bool SM>
__global__ void __maxnreg__(128) k_lu_panel(const LuProb<C>* __restrict__ P, int p, int ldp) {
  typedef typename real_of<C>::type R;
  typedef unsigned long long u64;
  namespace cg = cooperative_groups;
  constexpr int NW = LP_T / 32;
  extern __shared__ __align__(16) unsigned char lu_sm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const LuProb<C> pr = P[blockIdx.x / cs];
  const int m = pr.m;
  if (p >= m) return;   // the whole cluster leaves
  const int jb = min(MAXNB, m - p), mr = m - p;
  C* pan = SM ? reinterpret_cast<C*>(lu_sm) : pr.A + p + (size_t)p * pr.ld;
  const size_t ld = SM ? ldp : pr.ld;
  // by column parity: the CTAs' proposals (their rows in slots 0 .. 7) and the diagonal row (slot 8)
  __shared__ C s_slot[2][9][MAXNB];
  __shared__ u64 s_key[2][8];
  __shared__ unsigned s_krow[2][8];
  __shared__ u64 s_wk[NW];
  __shared__ unsigned s_wr[NW];
  __shared__ C s_inv[MAXNB];
  constexpr int GB = LP_GROUP<R>;
  __shared__ C s_ub[GB < MAXNB ? GB : 1][MAXNB];   // the group's pivot rows
  static_assert(NW == 8, "a warp writes to each CTA of the cluster");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nch = ((mr + 31) / 32 - rank + cs - 1) / cs;   // this CTA's chunks of 32 rows
  // chunk ch, lane i: row offset g from p, stored row
  auto row_g = [&](int ch) { return (ch * cs + rank) * 32 + lane; };
  auto row_s = [&](int ch) { return SM ? ch * 32 + lane : row_g(ch); };
  // few chunks: several warps share one, each with its residue of the columns
  const int q_n = nch <= 1 ? 8 : nch <= 2 ? 4 : nch <= 4 ? 2 : 1, slots = NW / q_n;
  const int slot = warp % slots, q = warp / slots;
  if (SM)
    for (int ch = warp; ch < nch; ch += NW)
      if (row_g(ch) < mr)
        for (int k = 0; k < jb; ++k) pan[row_s(ch) + k * ld] = pr.A[p + row_g(ch) + (size_t)(p + k) * pr.ld];
  cluster.sync();   // every CTA of the cluster runs before one writes to another
  u64 key = 0;
  unsigned krow = 0xFFFFFFFFu;
  auto propose = [&](C a, int g) {
    const R v = abs2(a);
    u64 k;
    if (sizeof(R) == 8) k = (u64)__double_as_longlong((double)v); else k = (u64)__float_as_uint((float)v);
    if (k > (sizeof(R) == 8 ? 0x7FF0000000000000ull : 0x7F800000ull)) k = 0;   // NaN
    if (k > key || (k == key && (unsigned)g < krow)) { key = k; krow = (unsigned)g; }
  };
  for (int ch = warp; ch < nch; ch += NW)
    if (row_g(ch) < mr) propose(pan[row_s(ch)], row_g(ch));
  auto pick = [&](u64& k, unsigned& r) {   // the largest key of the warp, the lowest row among equals
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
    const u64 best = ((u64)hi << 32) | lo;
    r = __reduce_min_sync(0xffffffffu, k == best ? r : 0xFFFFFFFFu);
    k = best;
  };
  for (int jj = 0; jj < jb; ++jj) {
    const int par = jj & 1;
    pick(key, krow);
    if (lane == 0) { s_wk[warp] = key; s_wr[warp] = krow; }
    __syncthreads();
    u64 ck = lane < NW ? s_wk[lane] : 0;
    unsigned cr = lane < NW ? s_wr[lane] : 0xFFFFFFFFu;
    pick(ck, cr);
    if (warp < cs) {   // this CTA's proposal to CTA `warp`
      if (ck > 0 && lane < jb) {
        const int g = (int)cr, ch = (g / 32 - rank) / cs;
        cluster.map_shared_rank(&s_slot[par][rank][0], warp)[lane] = pan[(SM ? ch * 32 + g % 32 : g) + lane * ld];
      }
      if (rank == 0 && lane < jb) cluster.map_shared_rank(&s_slot[par][8][0], warp)[lane] = pan[jj + lane * ld];
      if (lane == 0) {
        *cluster.map_shared_rank(&s_key[par][rank], warp) = ck;
        *cluster.map_shared_rank(&s_krow[par][rank], warp) = cr;
      }
    }
    cluster.sync();   // the proposals have arrived
    u64 wk = lane < cs ? s_key[par][lane] : 0;
    unsigned wr = lane < cs ? s_krow[par][lane] : 0xFFFFFFFFu;
    pick(wk, wr);
    const int piv = wk > 0 ? (int)wr : jj;                   // offset from p
    const int owner = (piv / 32) % cs;
    const C* u = wk > 0 ? s_slot[par][owner] : s_slot[par][8];   // the row of U
    if (warp == 1) {
      const C d = u[jj];
      const R d2 = abs2(d), ri = d2 > 0 ? (R)1 / d2 : (R)0;
      if (lane == 0) s_inv[jj] = mk(d.x * ri, -d.y * ri);
    } else if (warp == 2) {
      if (piv != jj && rank == owner && lane < jb) {
        const int ch = (piv / 32 - rank) / cs;
        pan[(SM ? ch * 32 + piv % 32 : piv) + lane * ld] = s_slot[par][8][lane];
      }
    } else if (warp == 3) {
      if (piv != jj && rank == 0 && lane < jb) pan[jj + lane * ld] = u[lane];
      if (rank == 0 && lane == 0) {
        pr.ipiv[p + jj] = p + piv;
        if (wk == 0 && *pr.info == 0) *pr.info = p + jj + 1;
      }
    } else if (GB < MAXNB && warp == 4 && lane < jb) {
      s_ub[jj % GB][lane] = u[lane];
    }
    const int s0 = jj / GB * GB, ge = min(jb, s0 + GB);   // the group's columns
    __syncthreads();
    const C inv = s_inv[jj];
    key = 0;
    krow = 0xFFFFFFFFu;
    for (int ch = slot; ch < nch; ch += slots) {
      const int g = row_g(ch);
      if (g <= jj || g >= mr) continue;
      C* row = pan + row_s(ch);
      const C l = row[jj * ld] * inv;
      int k = jj + 1 + (q - (jj + 1) % q_n + q_n) % q_n;   // the first column after jj of this residue
      if (k == jj + 1 && k < ge) {
        C a = row[k * ld];
        cfms(a, l, u[k]);
        row[k * ld] = a;
        propose(a, g);
        k += q_n;
      }
      for (; k + 3 * q_n < ge; k += 4 * q_n) {   // four columns in flight
        C a0 = row[k * ld], a1 = row[(k + q_n) * ld], a2 = row[(k + 2 * q_n) * ld], a3 = row[(k + 3 * q_n) * ld];
        cfms(a0, l, u[k]); cfms(a1, l, u[k + q_n]); cfms(a2, l, u[k + 2 * q_n]); cfms(a3, l, u[k + 3 * q_n]);
        row[k * ld] = a0; row[(k + q_n) * ld] = a1; row[(k + 2 * q_n) * ld] = a2; row[(k + 3 * q_n) * ld] = a3;
      }
      for (; k < ge; k += q_n) {
        C a = row[k * ld];
        cfms(a, l, u[k]);
        row[k * ld] = a;
      }
    }
    if constexpr (GB < MAXNB) {
      if (jj != ge - 1 || ge == jb) continue;
      if (warp == 0 && lane < jb - ge) {
        C a[GB];
#pragma unroll
        for (int i = 0; i < GB; ++i) a[i] = s_ub[i][ge + lane];
#pragma unroll
        for (int c = 0; c < GB - 1; ++c)
#pragma unroll
          for (int i = c + 1; i < GB; ++i) cfms(a[i], s_ub[i][s0 + c] * s_inv[s0 + c], a[c]);
#pragma unroll
        for (int i = 0; i < GB; ++i) {
          s_ub[i][ge + lane] = a[i];
          if (rank == 0) pan[s0 + i + (ge + lane) * ld] = a[i];
        }
      }
      __syncthreads();   // the rows of U, and the group's columns up to date
      for (int ch = slot; ch < nch; ch += slots) {
        const int g = row_g(ch);
        if (g < ge || g >= mr) continue;
        C* row = pan + row_s(ch);
        C l[GB];
#pragma unroll
        for (int i = 0; i < GB; ++i) l[i] = row[(s0 + i) * ld] * s_inv[s0 + i];
        for (int k = ge + (q - ge % q_n + q_n) % q_n; k < jb; k += q_n) {
          C sum = czero<C>();
#pragma unroll
          for (int i = 0; i < GB; ++i) cfma(sum, l[i], s_ub[i][k]);
          const C a = row[k * ld] - sum;
          row[k * ld] = a;
          if (k == ge) propose(a, g);
        }
      }
    }
  }
  __syncthreads();
  for (int ch = warp; ch < nch; ch += NW)
    if (row_g(ch) < mr)
      for (int k = 0; k < jb; ++k) {
        const C a = pan[row_s(ch) + k * ld];
        pr.A[p + row_g(ch) + (size_t)(p + k) * pr.ld] = row_g(ch) > k ? a * s_inv[k] : a;
      }
  cluster.sync();   // no CTA leaves while another may still read its proposal
}

// Row interchanges of the panel applied to every other column, then the unit
// lower triangular solve U12 = L11^{-1} A12 on the columns right of the panel.
// A warp per column.  The warp composes the panel's jb interchanges into a map
// over the rows they touch: lane i holds the panel row p + i and the i-th of
// the at most jb rows below the panel (row, and whose entry comes there).  The
// column's entries are gathered through it (the panel rows are contiguous:
// coalesced), the rows below written back, and the solve runs across the
// lanes, each lane's row taking its subtractions in ascending order.
template <typename C>
__global__ void __launch_bounds__(256) k_lu_swap_trsm(const LuProb<C>* __restrict__ P, int p) {
  static_assert(MAXNB == 32, "a lane per panel row");
  const LuProb<C> pr = P[blockIdx.y];
  const int m = pr.m;
  if (p >= m) return;
  const int jb = min(MAXNB, m - p);
  __shared__ C s_l[MAXNB][MAXNB + 1];
  C* A = pr.A;
  const size_t ld = pr.ld;
  const int lane = threadIdx.x & 31;
  const int j0 = blockIdx.x * (blockDim.x >> 5);
  if (j0 + (int)(blockDim.x >> 5) > p + jb)   // some column right of the panel
    for (int e = threadIdx.x; e < jb * jb; e += blockDim.x) s_l[e % jb][e / jb] = A[p + e % jb + (size_t)(p + e / jb) * ld];
  __syncthreads();
  const int j = j0 + (threadIdx.x >> 5);
  if (j >= m || (j >= p && j < p + jb)) return;   // whole warps leave together
  const int piv = lane < jb ? pr.ipiv[p + lane] : 0;
  int org = p + lane, row = -1, orow = -1, cnt = 0;
  for (int c = 0; c < jb; ++c) {
    const int r = __shfl_sync(0xffffffffu, piv, c), oc = __shfl_sync(0xffffffffu, org, c);
    if (r < p + jb) {
      const int o = __shfl_sync(0xffffffffu, org, r - p);
      if (lane == r - p) org = oc;
      if (lane == c) org = o;
    } else {
      const unsigned hit = __ballot_sync(0xffffffffu, row == r);
      const int s = hit ? __ffs(hit) - 1 : cnt++;
      if (!hit && lane == s) { row = r; orow = r; }
      const int o = __shfl_sync(0xffffffffu, orow, s);
      if (lane == s) orow = oc;
      if (lane == c) org = o;
    }
  }
  C* col = A + (size_t)j * ld;
  C v = lane < jb ? col[org] : czero<C>();
  const C below = lane < cnt ? col[orow] : czero<C>();
  __syncwarp();                                    // every read before any write
  if (lane < cnt) col[row] = below;
  if (j >= p + jb) {
    for (int q = 0; q < jb - 1; ++q) {
      const C vq = shfl_c(v, q);
      if (lane > q && lane < jb) cfms(v, s_l[lane][q], vq);
    }
  }
  if (lane < jb) col[p + lane] = v;
}

// Trailing update A22 -= L21 * U12 on the trailing columns [p+jb+lo, p+jb+hi)
// (all of them: lo = 0, hi >= m).  Every entry is the same sum whatever the
// column range, so a split update gives the same bits as the whole one.
template <typename C>
__global__ void __launch_bounds__(256) k_lu_update(const LuProb<C>* __restrict__ P, int p, int nb, int lo, int hi) {
  const LuProb<C> pr = P[blockIdx.y];
  const int m = pr.m;
  if (p >= m) return;
  const int jb = min(nb, m - p);
  const int mt = m - p - jb;
  if (mt <= 0) return;
  const int c0 = p + jb + lo, c1 = p + jb + min(hi, mt);
  if (c1 <= c0) return;
  const int tiles_m = (mt + TB - 1) / TB, tiles_n = (c1 - c0 + TB - 1) / TB;
  const int t = blockIdx.x;
  if (t >= tiles_m * tiles_n) return;
  C* A = pr.A;
  const size_t ld = pr.ld;
  C mone = mk((typename real_of<C>::type)-1, (typename real_of<C>::type)0);
  gemm_tile<C, true>(mt, c1 - c0, jb, A + (p + jb) + p * ld, pr.ld, A + p + c0 * ld, pr.ld,
               A + (p + jb) + c0 * ld, pr.ld, mone, mk((typename real_of<C>::type)1, (typename real_of<C>::type)0),
               0, t % tiles_m, t / tiles_m);
}

// ---- LU solve ----------------------------------------------------------------------

template <typename C>
__global__ void k_getrs_swap(const SolveProb<C>* __restrict__ P) {
  const SolveProb<C> pr = P[blockIdx.y];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= pr.nrhs) return;
  C* col = pr.B + (size_t)j * pr.ldb;
  for (int c = 0; c < pr.m; ++c) {
    int r = pr.ipiv[c];
    if (r != c) { C t = col[c]; col[c] = col[r]; col[r] = t; }
  }
}

// Row interchanges: thread 0 composes the m interchanges into one map in
// shared memory (position i receives original row src[i]); the CTA then
// gathers each of its right-hand sides through a shared-memory stage.
constexpr int SW_RHS = 32;   // right-hand sides per CTA
template <typename C>
__global__ void __launch_bounds__(256) k_getrs_swap_smem(const SolveProb<C>* __restrict__ P) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const SolveProb<C> pr = P[blockIdx.y];
  const int j0 = blockIdx.x * SW_RHS;
  if (j0 >= pr.nrhs) return;
  C* stage = reinterpret_cast<C*>(sm_raw);
  int* src = reinterpret_cast<int*>(stage + pr.m);
  for (int i = threadIdx.x; i < pr.m; i += blockDim.x) src[i] = i;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int c = 0; c < pr.m; ++c) {
      const int r = pr.ipiv[c];
      if (r != c) { const int t = src[c]; src[c] = src[r]; src[r] = t; }
    }
  __syncthreads();
  const int j1 = min(pr.nrhs, j0 + SW_RHS);
  for (int j = j0; j < j1; ++j) {
    C* col = pr.B + (size_t)j * pr.ldb;
    for (int i = threadIdx.x; i < pr.m; i += blockDim.x) stage[i] = col[src[i]];
    __syncthreads();
    for (int i = threadIdx.x; i < pr.m; i += blockDim.x) col[i] = stage[i];
    __syncthreads();
  }
}

// Diagonal block solve on rows [p, p+jb), jb <= 32: unit lower (lower=1) or
// upper.  The block is staged in shared memory; one warp per right-hand side,
// lane r holding row p+r, each solved entry broadcast by a shuffle.
// per: right-hand sides per CTA.  A warp's column is a chain of up to 31
// dependent multiply-adds, in FP64 2 us of its SM quarter: with few columns in
// the batch each warp takes one and each SM quarter one warp.
constexpr int DG_RHS = 32;   // the most right-hand sides per CTA (8 warps)
inline int diag_per(int nprob, int maxrhs, int sms) {
  return (long)nprob * ((maxrhs + 3) / 4) <= sms ? 4 : (long)nprob * ((maxrhs + 7) / 8) <= 2 * sms ? 8 : DG_RHS;
}
template <typename C>
__global__ void __launch_bounds__(256) k_getrs_diag(const SolveProb<C>* __restrict__ P, int p, int nb, int lower, int per) {
  typedef typename real_of<C>::type R;
  __shared__ C sa[32][33];
  const SolveProb<C> pr = P[blockIdx.y];
  if (p >= pr.m) return;
  const int jb = min(nb, pr.m - p);
  for (int e = threadIdx.x; e < jb * jb; e += blockDim.x) {
    const int r = e % jb, c = e / jb;
    sa[r][c] = pr.A[p + r + (size_t)(p + c) * pr.ld];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  // reciprocals of the diagonal, all lanes at once (the solve chain below
  // then multiplies instead of dividing: FP64 division is a long sequence)
  const C dinv = (!lower && lane < jb) ? cdiv(mk((R)1, (R)0), sa[lane][lane]) : czero<C>();
  const int j1 = min(pr.nrhs, (int)(blockIdx.x + 1) * per);
  for (int j = blockIdx.x * per + (threadIdx.x >> 5); j < j1; j += blockDim.x >> 5) {
    C* col = pr.B + (size_t)j * pr.ldb + p;
    C x = lane < jb ? col[lane] : czero<C>();
    if (lower) {
      for (int c = 0; c < jb - 1; ++c) {
        const C xc = shfl_c(x, c);
        if (lane > c && lane < jb) cfms(x, sa[lane][c], xc);
      }
    } else {
      for (int c = jb - 1; c >= 0; --c) {
        if (lane == c) x = x * dinv;
        const C xc = shfl_c(x, c);
        if (lane < c) cfms(x, sa[lane][c], xc);
      }
    }
    if (lane < jb) col[lane] = x;
  }
}

// Off-diagonal update: lower -> B[p+jb:m) -= L[p+jb:m, p:p+jb] B[p:p+jb);
//                      upper -> B[0:p)    -= U[0:p, p:p+jb]    B[p:p+jb).
template <typename C>
__global__ void __launch_bounds__(256) k_getrs_update(const SolveProb<C>* __restrict__ P, int p, int nb, int lower) {
  typedef typename real_of<C>::type R;
  const SolveProb<C> pr = P[blockIdx.y];
  if (p >= pr.m) return;
  const int jb = min(nb, pr.m - p);
  const int r0 = lower ? p + jb : 0;
  const int mt = lower ? pr.m - p - jb : p;
  if (mt <= 0 || pr.nrhs <= 0) return;
  const int tiles_m = (mt + TB - 1) / TB, tiles_n = (pr.nrhs + TB - 1) / TB;
  const int t = blockIdx.x;
  if (t >= tiles_m * tiles_n) return;
  const size_t ld = pr.ld;
  gemm_tile<C, true>(mt, pr.nrhs, jb, pr.A + r0 + p * ld, pr.ld, pr.B + p, pr.ldb, pr.B + r0, pr.ldb,
               mk((R)-1, (R)0), mk((R)1, (R)0), 0, t % tiles_m, t / tiles_m);
}

// One triangle of the LU solves of a batch of matrices, each with at most CHAIN_MAX_RHS
// right-hand sides, as ONE launch: every matrix is a chain of RS_NB-row
// blocks, one CTA per block and group of rg right-hand sides (the columns
// are independent chains; in FP64 a CTA's products and diagonal solve are
// bound by its SM's FP64 rate, so fewer columns per CTA shorten every link
// of the chain).  Each CTA takes a ticket from a counter and
// reads its (matrix, block) from items[ticket]; the items are ordered so that
// every block comes after the blocks it depends on (lower: by block index
// from the top, upper: by distance from the bottom), hence a CTA only ever
// waits on CTAs that took a smaller ticket and are already running: no
// co-residency is assumed.  A CTA subtracts the products of the blocks it
// depends on in their order, each as two interleaved sums and as soon as
// that block's flag is up, then solves its diagonal block as k_getrs_diag
// does, stores the result and raises its own flag: ~4 launches per block less
// on the critical path than the blocked solve.  With rg <= 4 the two sums of a
// product (even and odd terms) are taken by two threads and joined in the same
// order, so the bits do not depend on rg.  Every wait
// is bounded (TS_WAIT_NS); a wait that runs out sets *err and the shared
// abort word, and every CTA then leaves without writing.
// items[t] = (matrix, block, flag base of the matrix and group, group);
// sync: [0] ticket, [1] abort, [2, 2 + items) flags; zeroed before the launch.
// no_flag (failure-path tests): every CTA first waits, with a 1 ms bound, on
// `never`, which nothing sets.
constexpr long long TS_WAIT_NS = 2000000000ll;   // 2 s per wait
__device__ __forceinline__ unsigned long long ts_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int ts_load_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ts_store_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// G: dependencies taken per round.  A round loads the coefficient blocks of
// the next G dependencies together, waits for the first one's flag, adds
// the later ones whose flags are already up, loads their solved rows
// together and subtracts their products one by one in dependency order: a
// block that is behind the chain's front catches up with one pair of
// memory round trips per round instead of per dependency.
template <typename C, int G>
__global__ void __launch_bounds__(256) k_trsv_chain(const SolveProb<C>* __restrict__ P, const int4* __restrict__ items,
                                                    int nitems, int lower, int rg, int* sync, int* err,
                                                    const int* never, int no_flag) {
  typedef typename real_of<C>::type R;
  constexpr int NB = 32;
  __shared__ C sl[G][NB][NB + 1];   // the off-diagonal blocks of this round's dependencies, [col][row]
  __shared__ C sx[G][NB][8];        // their solved rows (this CTA's right-hand sides)
  __shared__ C sa[NB][NB + 1];      // the diagonal block
  __shared__ C s_odd[G][4][NB];     // rg <= 4: the odd-term sums
  __shared__ int s_t, s_stop, s_cnt;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_t = atomicAdd(&sync[0], 1);
    s_stop = 0;
    if (no_flag) {
      const unsigned long long t0 = ts_now();
      while (ts_load_acquire(never) == 0) {
        if (ts_load_acquire(&sync[1]) != 0) break;
        if ((long long)(ts_now() - t0) > 1000000ll) { atomicExch(err, 1); atomicExch(&sync[1], 1); break; }
        __nanosleep(64);
      }
      s_stop = 1;
    }
  }
  __syncthreads();
  if (s_stop) return;
  const int t = s_t;
  if (t >= nitems) return;
  const int4 it = items[t];
  const SolveProb<C> pr = P[it.x];
  const int m = pr.m;
  const int q0 = it.w * rg, nrhs = min(rg, pr.nrhs - q0);   // this CTA's columns q0 .. q0 + nrhs - 1
  if (nrhs <= 0) return;   // the whole (matrix, group) is empty: nobody waits on its flags
  const int nblk = (m + NB - 1) / NB;
  const int b = it.y;
  const int r0 = b * NB, jb = min(NB, m - r0);
  const size_t ld = pr.ld;
  int* flags = sync + 2 + it.z;
  for (int e = tid; e < jb * jb; e += 256) {
    const int r = e % jb, c = e / jb;
    sa[r][c] = pr.A[r0 + r + (size_t)(r0 + c) * ld];
  }
  // this thread's entry (row i, right-hand side q) of the block being solved;
  // with rg <= 4 thread h = 1 of (i, q) takes the odd-term sums for h = 0
  const bool split = rg <= 4;
  const int i = tid & 31, q = split ? (tid >> 5) % rg : tid >> 5, h = split ? (tid >> 5) / rg : 0;
  const bool mine = i < jb && q < nrhs && h == 0;
  const bool odd = split && i < jb && q < nrhs && h == 1;
  C x = mine ? pr.B[r0 + i + (size_t)(q0 + q) * pr.ldb] : czero<C>();
  const int ndep = lower ? b : nblk - 1 - b;
  auto dep = [&](int d) { return lower ? d : nblk - 1 - d; };   // the d-th block this one depends on
  for (int d0 = 0; d0 < ndep;) {
    const int gmax = min(G, ndep - d0);
    // the coefficients do not depend on the flags: load them first
    for (int g = 0; g < gmax; ++g) {
      const int c0 = dep(d0 + g) * NB, jbj = min(NB, m - c0);
      for (int e = tid; e < jb * jbj; e += 256) {
        const int r = e % jb, c = e / jb;
        sl[g][c][r] = pr.A[r0 + r + (size_t)(c0 + c) * ld];
      }
    }
    if (tid == 0) {
      const unsigned long long t0 = ts_now();
      while (ts_load_acquire(&flags[dep(d0)]) == 0) {
        if (ts_load_acquire(&sync[1]) != 0) { s_stop = 1; break; }
        if ((long long)(ts_now() - t0) > TS_WAIT_NS) {
          atomicExch(err, 1);
          atomicExch(&sync[1], 1);
          s_stop = 1;
          break;
        }
        __nanosleep(64);
      }
      int cnt = 1;
      while (cnt < gmax && ts_load_acquire(&flags[dep(d0 + cnt)]) != 0) ++cnt;
      s_cnt = cnt;
    }
    __syncthreads();
    if (s_stop) return;
    const int cnt = s_cnt;
    for (int g = 0; g < cnt; ++g) {
      const int c0 = dep(d0 + g) * NB, jbj = min(NB, m - c0);
      for (int e = tid; e < jbj * nrhs; e += 256) {
        const int l = e % jbj, qq = e / jbj;
        sx[g][l][qq] = __ldcg(pr.B + c0 + l + (size_t)(q0 + qq) * pr.ldb);
      }
    }
    __syncthreads();
    for (int g = 0; g < cnt; ++g) {
      const int jbj = min(NB, m - dep(d0 + g) * NB);
      if (split) {
        // acc0 over the even terms, acc1 over the odd ones, each in order
        C acc = czero<C>();
        if (mine || odd)
          for (int l = h; l < jbj; l += 2) cfma(acc, sl[g][l][i], sx[g][l][q]);
        if (odd) s_odd[g][q][i] = acc;
        __syncthreads();
        if (mine) x = x - (acc + s_odd[g][q][i]);
      } else if (mine) {
        C acc0 = czero<C>(), acc1 = czero<C>();
        int l = 0;
        for (; l + 1 < jbj; l += 2) {
          cfma(acc0, sl[g][l][i], sx[g][l][q]);
          cfma(acc1, sl[g][l + 1][i], sx[g][l + 1][q]);
        }
        if (l < jbj) cfma(acc0, sl[g][l][i], sx[g][l][q]);
        x = x - (acc0 + acc1);
      }
    }
    __syncthreads();   // sl, sx and s_odd are refilled next
    d0 += cnt;
  }
  // the diagonal block: warp q solves right-hand side q, lane r holds row r
  if (mine) sx[0][i][q] = x;
  __syncthreads();
  if (warp < nrhs) {
    const C dinv = (!lower && lane < jb) ? cdiv(mk((R)1, (R)0), sa[lane][lane]) : czero<C>();
    C y = lane < jb ? sx[0][lane][warp] : czero<C>();
    if (lower) {
      for (int c = 0; c < jb - 1; ++c) {
        const C yc = shfl_c(y, c);
        if (lane > c && lane < jb) cfms(y, sa[lane][c], yc);
      }
    } else {
      for (int c = jb - 1; c >= 0; --c) {
        if (lane == c) y = y * dinv;
        const C yc = shfl_c(y, c);
        if (lane < c) cfms(y, sa[lane][c], yc);
      }
    }
    if (lane < jb) pr.B[r0 + lane + (size_t)(q0 + warp) * pr.ldb] = y;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) ts_store_release(&flags[b], 1);
}

// Products with at most GEMV_MAX_N columns (solves for one to three waves).
// A 32 x 32 tile left 29 to 31 of its columns empty, FP64 operations and all;
// here a CTA takes 32 rows, its 8 warps every eighth term of the sums, a lane
// a row, so that A is read once, 512 bytes at a time, and only the products
// themselves are formed.  The warps' sums meet in a fixed order.
template <typename C, int N>
__device__ __forceinline__ void gemv_rows(const GemmDesc<C>& g, int r0, C (*red)[32][GEMV_MAX_N]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, row = r0 + lane;
  C acc[N];
#pragma unroll
  for (int j = 0; j < N; ++j) acc[j] = czero<C>();
  if (row < g.m) {
#pragma unroll 4
    for (int l = warp; l < g.k; l += 8) {
      const C a = g.A[row + (size_t)l * g.lda];
#pragma unroll
      for (int j = 0; j < N; ++j) cfma(acc[j], a, g.B[l + (size_t)j * g.ldb]);
    }
  }
#pragma unroll
  for (int j = 0; j < N; ++j) red[warp][lane][j] = acc[j];
  __syncthreads();
  if (warp < N && row < g.m) {
    C v = red[0][lane][warp];
#pragma unroll
    for (int w = 1; w < 8; ++w) v = v + red[w][lane][warp];
    C* p = g.Cm + row + (size_t)warp * g.ldc;
    v = g.alpha * v;
    if (!g.beta_zero) v = v + g.beta * (*p);
    *p = v;
  }
}

template <typename C>
__global__ void __launch_bounds__(256) k_gemv_batched(const GemmDesc<C>* __restrict__ d,
                                                      const int* __restrict__ tile_off, int nprob) {
  __shared__ C red[8][32][GEMV_MAX_N];
  const int t = blockIdx.x;
  int lo = 0, hi = nprob;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tile_off[mid] <= t) lo = mid; else hi = mid;
  }
  const GemmDesc<C> g = d[lo];
  const int r0 = (t - tile_off[lo]) * 32;
  if (g.n == 1) gemv_rows<C, 1>(g, r0, red);
  else if (g.n == 2) gemv_rows<C, 2>(g, r0, red);
  else gemv_rows<C, 3>(g, r0, red);
}

}  // namespace

template <typename C>
void la_gemv_batched(const GemmDesc<C>* d_desc, const int* d_tile_off, int nprob, int total_tiles, cudaStream_t st) {
  if (nprob <= 0 || total_tiles <= 0) return;
  KPROF_BEGIN(st);
  k_gemv_batched<C><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob);
  pm_launch_count_add(1);
  KPROF_END(st, kname<C>("gemv_batched", "gemv_batched32"), 0.0);
}

template <typename C>
void la_gemm_batched(const GemmDesc<C>* d_desc, const int* d_tile_off, int nprob, int total_tiles,
                     cudaStream_t st) {
  if (nprob <= 0 || total_tiles <= 0) return;
  KPROF_BEGIN(st);
  k_gemm_batched<C><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob);
  pm_launch_count_add(1);
  KPROF_END(st, kname<C>("gemm_batched", "gemm_batched32"), 0.0);
}

const GemmShape kGemmShapes[GEMM_NSHAPES] = {{32, 32}, {64, 64}, {64, 32}, {128, 8}, {64, 16}};

template <typename C>
void la_gemm_batched_shape(int shape, const GemmDesc<C>* d_desc, const int* d_tile_off, int nprob, int total_tiles,
                           cudaStream_t st) {
  if (nprob <= 0 || total_tiles <= 0) return;
  KPROF_BEGIN(st);
  switch (shape) {
    case 1: k_gemm_batched_t<C, 64, 64, 4, 4><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob); break;
    case 2: k_gemm_batched_t<C, 64, 32, 4, 2><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob); break;
    case 3: k_gemm_batched_t<C, 128, 8, 4, 1><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob); break;
    case 4: k_gemm_batched_t<C, 64, 16, 2, 2><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob); break;
    default: k_gemm_batched<C><<<total_tiles, 256, 0, st>>>(d_desc, d_tile_off, nprob); break;
  }
  pm_launch_count_add(1);
  KPROF_END(st, kname<C>("gemm_batched", "gemm_batched32"), 0.0);
}

constexpr int LU_NB = MAXNB;
constexpr size_t LU_PANEL_SMEM = 216 * 1024;   // a CTA's rows of a panel up to this size stay in shared memory
constexpr int RS_NB = 32;

// Flop counts of step p (panel, unit-lower solve of U12, trailing GEMM) for the profiler.
inline void lu_step_flops(const int* h_m, int nprob, int p, double& fp, double& fs, double& fu) {
  fp = fs = fu = 0;
  for (int i = 0; i < nprob; ++i) {
    const int m = h_m[i];
    if (p >= m) continue;
    const double jb = std::min(LU_NB, m - p), rest = m - p - jb, h = m - p;
    fp += 8.0 * (h * jb * jb / 2);
    fs += 8.0 * rest * jb * jb / 2;
    fu += 8.0 * rest * rest * jb;
  }
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Panel of step p: as many CTAs per matrix (up to 8) as fill the SMs, but no
// more than chunks of 32 rows, and as many as keep the rows in shared memory.
template <typename C>
void lu_panel(const LuProb<C>* d_prob, int nprob, int maxm, int p, cudaStream_t st) {
  const int sms = sm_count(), nch = (maxm - p + 31) / 32;
  auto bytes = [&](int cs) { return (size_t)((nch + cs - 1) / cs) * 32 * LU_NB * sizeof(C); };
  int cs = 1;
  while (cs < 8 && cs < nch && ((long)nprob * cs * 2 <= sms || bytes(cs) > LU_PANEL_SMEM)) cs *= 2;
  const bool smem = bytes(cs) <= LU_PANEL_SMEM;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nprob * cs);
  cfg.blockDim = dim3(LP_T);
  cfg.dynamicSmemBytes = smem ? bytes(cs) : 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int ldp = ((nch + cs - 1) / cs) * 32;
  if (smem) {
    // the same value every time: idempotent across threads and devices
    cudaFuncSetAttribute(k_lu_panel<C, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LU_PANEL_SMEM);
    cudaLaunchKernelEx(&cfg, k_lu_panel<C, true>, d_prob, p, ldp);
  } else {
    cudaLaunchKernelEx(&cfg, k_lu_panel<C, false>, d_prob, p, ldp);
  }
}

// The trailing update of step p on trailing columns [lo, hi): complex128 on
// the tensor cores, complex64 on the FP32 pipe.
template <typename C>
void lu_update(const LuProb<C>* d_prob, int nprob, int maxm, int p, int lo, int hi, cudaStream_t st) {
  const int mt = maxm - p - LU_NB, n = std::min(hi, mt) - lo;
  if constexpr (std::is_same<C, double2>::value) oz_lu_update(d_prob, nprob, maxm, p, LU_NB, lo, hi, oz_err_word(), st);
  else k_lu_update<C><<<dim3(((mt + TB - 1) / TB) * ((n + TB - 1) / TB), nprob), 256, 0, st>>>(d_prob, p, LU_NB, lo, hi);
}

// The off-diagonal update of a blocked triangular solve, by the same rule.
template <typename C>
void getrs_update(const SolveProb<C>* d_prob, int nprob, int maxm, int maxrhs, int p, int lower, cudaStream_t st) {
  const int mt = lower ? maxm - p - RS_NB : p;
  if constexpr (std::is_same<C, double2>::value)
    oz_getrs_update(d_prob, nprob, maxm, maxrhs, p, RS_NB, lower, oz_err_word(), st);
  else
    k_getrs_update<C><<<dim3(((mt + TB - 1) / TB) * ((maxrhs + TB - 1) / TB), nprob), 256, 0, st>>>(d_prob, p, RS_NB, lower);
}

// A few large matrices (the top-level LU) with look-ahead: step p's update
// of the next panel's LU_NB columns runs first, on a high-priority stream
// with the panels, and the rest of the trailing update on a low-priority
// stream, so that panel p+1 (latency-bound, on one 8-CTA cluster) overlaps
// the bulk of update p instead of leaving the other SMs idle.  Step p+1's
// interchanges wait for that update.  The kernels and their arithmetic are
// those of the plain sequence (identical bits).
template <typename C>
void la_getrf_lookahead(const LuProb<C>* d_prob, int nprob, int maxm, const int* h_m, cudaStream_t st) {
  int pr_lo = 0, pr_hi = 0;
  cudaDeviceGetStreamPriorityRange(&pr_lo, &pr_hi);
  cudaStream_t sp = nullptr, su = nullptr;
  cudaStreamCreateWithPriority(&sp, cudaStreamNonBlocking, pr_hi);
  cudaStreamCreateWithPriority(&su, cudaStreamNonBlocking, pr_lo);
  cudaEvent_t e_fork, e_next, e_rest;
  cudaEventCreateWithFlags(&e_fork, cudaEventDisableTiming);
  cudaEventCreateWithFlags(&e_next, cudaEventDisableTiming);
  cudaEventCreateWithFlags(&e_rest, cudaEventDisableTiming);
  cudaEventRecord(e_fork, st);
  cudaStreamWaitEvent(sp, e_fork, 0);
  cudaStreamWaitEvent(su, e_fork, 0);
  bool rest_pending = false;
  for (int p = 0; p < maxm; p += LU_NB) {
    double fp, fs, fu;
    lu_step_flops(h_m, nprob, p, fp, fs, fu);
    KPROF_BEGIN(sp);
    lu_panel<C>(d_prob, nprob, maxm, p, sp);
    pm_launch_count_add(1);
    KPROF_END(sp, kname<C>("lu_panel", "lu_panel32"), fp);
    if (rest_pending) cudaStreamWaitEvent(sp, e_rest, 0);
    dim3 g1((maxm + 7) / 8, nprob);   // a warp per column
    KPROF_BEGIN(sp);
    k_lu_swap_trsm<C><<<g1, 256, 0, sp>>>(d_prob, p);
    pm_launch_count_add(1);
    KPROF_END(sp, kname<C>("lu_swap_trsm", "lu_swap_trsm32"), fs);
    rest_pending = false;
    const int mt = maxm - p - LU_NB;
    if (mt <= 0) continue;
    const int nrest = mt - LU_NB;
    if (nrest > 0) cudaEventRecord(e_next, sp);   // interchanges and U12 of step p are done
    const double fn = fu * std::min(1.0, (double)LU_NB / mt);
    KPROF_BEGIN(sp);
    lu_update<C>(d_prob, nprob, maxm, p, 0, LU_NB, sp);
    pm_launch_count_add(1);
    KPROF_END(sp, kname<C>("lu_update", "lu_update32"), fn);
    if (nrest > 0) {
      cudaStreamWaitEvent(su, e_next, 0);
      KPROF_BEGIN(su);
      lu_update<C>(d_prob, nprob, maxm, p, LU_NB, 1 << 30, su);
      pm_launch_count_add(1);
      KPROF_END(su, kname<C>("lu_update", "lu_update32"), fu - fn);
      cudaEventRecord(e_rest, su);
      rest_pending = true;
    }
  }
  cudaEventRecord(e_next, sp);
  cudaEventRecord(e_rest, su);
  cudaStreamWaitEvent(st, e_next, 0);
  cudaStreamWaitEvent(st, e_rest, 0);
  cudaEventDestroy(e_fork);
  cudaEventDestroy(e_next);
  cudaEventDestroy(e_rest);
  cudaStreamDestroy(sp);
  cudaStreamDestroy(su);
}

template <typename C>
void la_getrf_batched(const LuProb<C>* d_prob, int nprob, int maxm, const int* h_m, cudaStream_t st) {
  if (nprob <= 0 || maxm <= 0) return;
  if (nprob <= 8 && maxm >= 512) {
    la_getrf_lookahead<C>(d_prob, nprob, maxm, h_m, st);
    return;
  }
  for (int p = 0; p < maxm; p += LU_NB) {
    double fp = 0, fs = 0, fu = 0;
    if (g_kprof) lu_step_flops(h_m, nprob, p, fp, fs, fu);
    KPROF_BEGIN(st);
    lu_panel<C>(d_prob, nprob, maxm, p, st);
    pm_launch_count_add(1);
    KPROF_END(st, kname<C>("lu_panel", "lu_panel32"), fp);
    dim3 g1((maxm + 7) / 8, nprob);   // a warp per column
    KPROF_BEGIN(st);
    k_lu_swap_trsm<C><<<g1, 256, 0, st>>>(d_prob, p);
    pm_launch_count_add(1);
    KPROF_END(st, kname<C>("lu_swap_trsm", "lu_swap_trsm32"), fs);
    int mt = maxm - p - LU_NB;
    if (mt > 0) {
      KPROF_BEGIN(st);
      lu_update<C>(d_prob, nprob, maxm, p, 0, 1 << 30, st);
      pm_launch_count_add(1);
      KPROF_END(st, kname<C>("lu_update", "lu_update32"), fu);
    }
  }
}

int la_chain_items(const int* h_m, int nprob, int groups, std::vector<int4>& items) {
  std::vector<int> nb(nprob), base(nprob);
  int total = 0, maxb = 0;
  for (int i = 0; i < nprob; ++i) {
    nb[i] = std::max(0, (h_m[i] + RS_NB - 1) / RS_NB);
    base[i] = total;
    total += nb[i];
    maxb = std::max(maxb, nb[i]);
  }
  items.clear();
  items.reserve(2 * (size_t)total * groups);
  // flags of (matrix i, group g): groups * base[i] + g * nb[i] + block
  for (int d = 0; d < maxb; ++d)   // lower: block d of every matrix that has one
    for (int i = 0; i < nprob; ++i)
      for (int g = 0; g < groups; ++g)
        if (d < nb[i]) items.push_back(make_int4(i, d, groups * base[i] + g * nb[i], g));
  for (int d = 0; d < maxb; ++d)   // upper: block d from the bottom
    for (int i = 0; i < nprob; ++i)
      for (int g = 0; g < groups; ++g)
        if (d < nb[i]) items.push_back(make_int4(i, nb[i] - 1 - d, groups * base[i] + g * nb[i], g));
  return total * groups;
}
int la_chain_sync_ints(int total) { return 2 * (2 + total) + 1; }

template <typename C>
void la_getrs_batched(const SolveProb<C>* d_prob, int nprob, int maxm, int maxrhs, const int* h_m,
                      const int* h_rhs, cudaStream_t st, const ChainArgs* chain) {
  if (nprob <= 0 || maxm <= 0 || maxrhs <= 0) return;
  double fl = 0;
  if (g_kprof)
    for (int i = 0; i < nprob; ++i) fl += 8.0 * (double)h_m[i] * h_m[i] * h_rhs[i];
  KPROF_BEGIN(st);
  const size_t swap_smem = (size_t)maxm * (sizeof(C) + sizeof(int));
  if (swap_smem <= 200 * 1024) {
    // the same value every time: idempotent across threads and devices
    if (swap_smem > 48 * 1024)
      cudaFuncSetAttribute(k_getrs_swap_smem<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    k_getrs_swap_smem<C><<<dim3((maxrhs + SW_RHS - 1) / SW_RHS, nprob), 256, swap_smem, st>>>(d_prob);
  } else {
    dim3 gsw((maxrhs + 127) / 128, nprob);
    k_getrs_swap<C><<<gsw, 128, 0, st>>>(d_prob);
  }
  pm_launch_count_add(1);
  if (chain && maxrhs <= CHAIN_MAX_RHS) {
    // few right-hand sides: each triangle of every matrix in one chained launch
    const int T = chain->total_blocks;
    cudaMemsetAsync(chain->sync, 0, sizeof(int) * la_chain_sync_ints(T), st);
    const int* never = chain->sync + 2 * (2 + T);
    if (T > 0) {
      // complex64: three dependencies per round; FP64: one (its products are
      // bound by the SM's FP64 rate, not by the round trips)
      constexpr int G = sizeof(C) == sizeof(double2) ? 1 : 3;
      k_trsv_chain<C, G><<<T, 256, 0, st>>>(d_prob, chain->items, T, 1, chain->rhs_per_cta, chain->sync, chain->err,
                                            never, chain->no_flag);
      k_trsv_chain<C, G><<<T, 256, 0, st>>>(d_prob, chain->items + T, T, 0, chain->rhs_per_cta, chain->sync + 2 + T,
                                            chain->err, never, chain->no_flag);
      pm_launch_count_add(2);
    }
    KPROF_END(st, kname<C>("getrs", "getrs32"), fl);
    return;
  }
  const int per = diag_per(nprob, maxrhs, sm_count());
  const dim3 gs((maxrhs + per - 1) / per, nprob);
  const int dt = std::min(256, 32 * per);
  for (int p = 0; p < maxm; p += RS_NB) {
    k_getrs_diag<C><<<gs, dt, 0, st>>>(d_prob, p, RS_NB, 1, per);
    pm_launch_count_add(1);
    if (maxm - p - RS_NB > 0) {
      getrs_update<C>(d_prob, nprob, maxm, maxrhs, p, 1, st);
      pm_launch_count_add(1);
    }
  }
  for (int p = ((maxm - 1) / RS_NB) * RS_NB; p >= 0; p -= RS_NB) {
    k_getrs_diag<C><<<gs, dt, 0, st>>>(d_prob, p, RS_NB, 0, per);
    pm_launch_count_add(1);
    if (p > 0) {
      getrs_update<C>(d_prob, nprob, maxm, maxrhs, p, 0, st);
      pm_launch_count_add(1);
    }
  }
  KPROF_END(st, kname<C>("getrs", "getrs32"), fl);
}

template <typename C>
void la_trsm_upper_batched(const SolveProb<C>* d_prob, int nprob, int maxm, int maxrhs, const char* name,
                           double flops, cudaStream_t st) {
  if (nprob <= 0 || maxm <= 0 || maxrhs <= 0) return;
  KPROF_BEGIN(st);
  const int per = diag_per(nprob, maxrhs, sm_count());
  const dim3 gs((maxrhs + per - 1) / per, nprob);
  const int dt = std::min(256, 32 * per);
  int last = ((maxm - 1) / RS_NB) * RS_NB;
  for (int p = last; p >= 0; p -= RS_NB) {
    k_getrs_diag<C><<<gs, dt, 0, st>>>(d_prob, p, RS_NB, 0, per);
    pm_launch_count_add(1);
    if (p > 0) {
      getrs_update<C>(d_prob, nprob, maxm, maxrhs, p, 0, st);
      pm_launch_count_add(1);
    }
  }
  KPROF_END(st, name, flops);
}

template void la_trsm_upper_batched<double2>(const SolveProb<double2>*, int, int, int, const char*, double,
                                             cudaStream_t);
template void la_trsm_upper_batched<float2>(const SolveProb<float2>*, int, int, int, const char*, double,
                                            cudaStream_t);
template void la_gemm_batched_shape<double2>(int, const GemmDesc<double2>*, const int*, int, int, cudaStream_t);
template void la_gemm_batched_shape<float2>(int, const GemmDesc<float2>*, const int*, int, int, cudaStream_t);
template void la_gemv_batched<double2>(const GemmDesc<double2>*, const int*, int, int, cudaStream_t);
template void la_gemv_batched<float2>(const GemmDesc<float2>*, const int*, int, int, cudaStream_t);
template void la_gemm_batched<double2>(const GemmDesc<double2>*, const int*, int, int, cudaStream_t);
template void la_gemm_batched<float2>(const GemmDesc<float2>*, const int*, int, int, cudaStream_t);
template void la_getrf_batched<double2>(const LuProb<double2>*, int, int, const int*, cudaStream_t);
template void la_getrf_batched<float2>(const LuProb<float2>*, int, int, const int*, cudaStream_t);
template void la_getrs_batched<double2>(const SolveProb<double2>*, int, int, int, const int*, const int*, cudaStream_t,
                                        const ChainArgs*);
template void la_getrs_batched<float2>(const SolveProb<float2>*, int, int, int, const int*, const int*, cudaStream_t,
                                       const ChainArgs*);
