// FP64-accurate tensor-core products (oz.cuh) for the batched GEMMs and the
// trailing updates of the FP64 LU and LU solves.
#include "oz_gemm.cuh"
#include "oz.cuh"
#include "prof.cuh"
#include <algorithm>

thread_local int* g_oz_err = nullptr;
thread_local int g_oz_no_arrive = 0;

namespace {

// C (m x n) := combine(C, A B) on the row tile r0 and the column tiles [t0, t1).
// MODE 0: alpha A B + beta C (beta_zero: C not read); 1: C - A B.
template <int MODE>
__device__ __forceinline__ void oz_tiles_of(oz::Cta& cta, int m, int n, int k, const double2* __restrict__ A, size_t lda,
                                            const double2* __restrict__ B, size_t ldb, double2* C, size_t ldc, int r0,
                                            int t0, int t1, double2 alpha, double2 beta, int beta_zero) {
  const int warp = threadIdx.x >> 5, row = r0 + 32 * (warp & 3) + (threadIdx.x & 31), cg = 8 * (warp >> 2);
  for (int t = t0; t < t1; ++t) {
    const int c0 = t * oz::TN;
    double2 v[8];   // MODE 0: the sums; 1: C, loaded during the first stage's MMAs, minus them
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = make_double2(0.0, 0.0);
    for (int l0 = 0; l0 < k; l0 += oz::TKC)
      oz::stage(cta, k > oz::TKC || t == t0,
                [&](int i, int l) {
                  return r0 + i < m && l0 + l < k ? A[r0 + i + (l0 + l) * lda] : make_double2(0.0, 0.0);
                },
                [&](int l, int j) {
                  return l0 + l < k && c0 + j < n ? B[l0 + l + (c0 + j) * ldb] : make_double2(0.0, 0.0);
                },
                [&](int j, int part, double d) {
                  double& o = part == 0 ? v[j].x : v[j].y;
                  o = MODE == 1 ? o - d : o + d;
                },
                [&] {
                  if (MODE != 1 || l0 > 0 || row >= m) return;
#pragma unroll
                  for (int j = 0; j < 8; ++j)
                    if (c0 + cg + j < n) v[j] = C[row + (c0 + cg + j) * ldc];
                });
    if (row < m && cta.ok) {
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (c0 + cg + j < n) {
          double2* p = C + row + (c0 + cg + j) * ldc;
          if (MODE == 0) {
            if (!(alpha.y == 0.0 && alpha.x == 1.0)) v[j] = alpha * v[j];
            if (!beta_zero) v[j] = v[j] + beta * (*p);
          }
          *p = v[j];
        }
    }
  }
}

__global__ void __launch_bounds__(oz::T) k_oz_gemm(const GemmDesc<double2>* __restrict__ d, const int* __restrict__ off,
                                                   int nprob, int per, int* err, int no_arrive) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const int t = blockIdx.x;
  int lo = 0, hi = nprob;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= t) lo = mid; else hi = mid;
  }
  const GemmDesc<double2> g = d[lo];
  const int local = t - off[lo], tm = (g.m + oz::TM - 1) / oz::TM, tn = (g.n + oz::TN - 1) / oz::TN;
  const int r0 = (local % tm) * oz::TM, t0 = (local / tm) * per;
  oz::Cta cta = oz::begin(sm, no_arrive);
  if (g.alpha.x == -1.0 && g.alpha.y == 0.0 && g.beta.x == 1.0 && g.beta.y == 0.0 && !g.beta_zero)
    oz_tiles_of<1>(cta, g.m, g.n, g.k, g.A, g.lda, g.B, g.ldb, g.Cm, g.ldc, r0, t0, min(tn, t0 + per), g.alpha, g.beta, 0);
  else
    oz_tiles_of<0>(cta, g.m, g.n, g.k, g.A, g.lda, g.B, g.ldb, g.Cm, g.ldc, r0, t0, min(tn, t0 + per), g.alpha, g.beta,
                   g.beta_zero);
  oz::end(cta, err);
}

__global__ void __launch_bounds__(oz::T) k_oz_lu_update(const LuProb<double2>* __restrict__ P, int p, int nb, int lo, int hi,
                                                        int per, int* err, int no_arrive) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const LuProb<double2> pr = P[blockIdx.z];
  if (p >= pr.m) return;
  const int jb = min(nb, pr.m - p), mt = pr.m - p - jb;
  const int c0 = p + jb + lo, n = p + jb + min(hi, mt) - c0;
  const int r0 = blockIdx.x * oz::TM, t0 = blockIdx.y * per, tn = (n + oz::TN - 1) / oz::TN;
  if (r0 >= mt || t0 >= tn) return;
  const size_t ld = pr.ld;
  const double2 z = make_double2(0.0, 0.0);
  oz::Cta cta = oz::begin(sm, no_arrive);
  oz_tiles_of<1>(cta, mt, n, jb, pr.A + (p + jb) + p * ld, ld, pr.A + p + c0 * ld, ld, pr.A + (p + jb) + c0 * ld, ld, r0, t0,
                 min(tn, t0 + per), z, z, 0);
  oz::end(cta, err);
}

__global__ void __launch_bounds__(oz::T) k_oz_getrs_update(const SolveProb<double2>* __restrict__ P, int p, int nb, int lower,
                                                           int per, int* err, int no_arrive) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const SolveProb<double2> pr = P[blockIdx.z];
  if (p >= pr.m) return;
  const int jb = min(nb, pr.m - p);
  const int b0 = lower ? p + jb : 0, mt = lower ? pr.m - p - jb : p;
  const int r0 = blockIdx.x * oz::TM, t0 = blockIdx.y * per, tn = (pr.nrhs + oz::TN - 1) / oz::TN;
  if (r0 >= mt || t0 >= tn) return;
  const double2 z = make_double2(0.0, 0.0);
  oz::Cta cta = oz::begin(sm, no_arrive);
  oz_tiles_of<1>(cta, mt, pr.nrhs, jb, pr.A + b0 + p * (size_t)pr.ld, pr.ld, pr.B + p, pr.ldb, pr.B + b0, pr.ldb, r0, t0,
                 min(tn, t0 + per), z, z, 0);
  oz::end(cta, err);
}

}  // namespace

int oz_per(long tiles) { return (int)std::max(1l, std::min(8l, tiles / 304)); }

void oz_gemm_batched(const GemmDesc<double2>* d_desc, const int* d_off, int nprob, int total, int per, int* err,
                     cudaStream_t st) {
  if (nprob <= 0 || total <= 0) return;
  KPROF_BEGIN(st);
  // the same value every time: idempotent across threads and devices
  cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM);
  k_oz_gemm<<<total, oz::T, oz::SMEM, st>>>(d_desc, d_off, nprob, per, err, g_oz_no_arrive);
  pm_launch_count_add(1);
  KPROF_END(st, "gemm_oz", 0.0);
}

void oz_lu_update(const LuProb<double2>* d_prob, int nprob, int maxm, int p, int nb, int lo, int hi, int* err,
                  cudaStream_t st) {
  const int mt = maxm - p - nb, n = std::min(hi, mt) - lo;
  if (nprob <= 0 || mt <= 0 || n <= 0) return;
  const int tm = (mt + oz::TM - 1) / oz::TM, tn = (n + oz::TN - 1) / oz::TN, per = oz_per((long)tm * tn * nprob);
  cudaFuncSetAttribute(k_oz_lu_update, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM);
  k_oz_lu_update<<<dim3(tm, (tn + per - 1) / per, nprob), oz::T, oz::SMEM, st>>>(d_prob, p, nb, lo, hi, per, err,
                                                                                 g_oz_no_arrive);
}

void oz_getrs_update(const SolveProb<double2>* d_prob, int nprob, int maxm, int maxrhs, int p, int nb, int lower, int* err,
                     cudaStream_t st) {
  const int mt = lower ? maxm - p - nb : p;
  if (nprob <= 0 || mt <= 0 || maxrhs <= 0) return;
  const int tm = (mt + oz::TM - 1) / oz::TM, tn = (maxrhs + oz::TN - 1) / oz::TN, per = oz_per((long)tm * tn * nprob);
  cudaFuncSetAttribute(k_oz_getrs_update, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM);
  k_oz_getrs_update<<<dim3(tm, (tn + per - 1) / per, nprob), oz::T, oz::SMEM, st>>>(d_prob, p, nb, lower, per, err,
                                                                                    g_oz_no_arrive);
}
