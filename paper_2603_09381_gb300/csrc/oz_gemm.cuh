// Launchers of the FP64-accurate tensor-core products (oz.cuh): batched GEMM
// and the trailing updates of the FP64 LU and LU solves.
#pragma once
#include "dense_la.cuh"
#include <stdexcept>

// Error word of the bounded tensor-core waits of the running call (device
// int, set to 1 when a wait runs out): thread-local, set by OzErrScope.
// no_arrive (tests of the timeout path): see oz::begin.
extern thread_local int* g_oz_err;
extern thread_local int g_oz_no_arrive;
struct OzErrScope {
  int* prev;
  int prev_no_arrive;
  explicit OzErrScope(int* e, bool no_arrive = false) : prev(g_oz_err), prev_no_arrive(g_oz_no_arrive) {
    g_oz_err = e;
    g_oz_no_arrive = no_arrive;
  }
  ~OzErrScope() {
    g_oz_err = prev;
    g_oz_no_arrive = prev_no_arrive;
  }
  OzErrScope(const OzErrScope&) = delete;
  OzErrScope& operator=(const OzErrScope&) = delete;
};
inline int* oz_err_word() {
  if (!g_oz_err) throw std::logic_error("FP64 tensor-core product without an error word");
  return g_oz_err;
}

// Tiles of an m x n product: rows in 128s, columns in groups of `per` tiles of 32.
inline int oz_tiles(int m, int n, int per) { return ((m + 127) / 128) * ((n + 32 * per - 1) / (32 * per)); }
// Column tiles per CTA for a batch of `tiles` single-tile products (A's digits are reused across them).
int oz_per(long tiles);

// d_off: prefix sums of oz_tiles(m, n, per).
void oz_gemm_batched(const GemmDesc<double2>* d_desc, const int* d_off, int nprob, int total, int per, int* err,
                     cudaStream_t st);
// A22 -= L21 U12 on trailing columns [p + jb + lo, p + jb + hi) of every matrix (k_lu_update's contract).
void oz_lu_update(const LuProb<double2>* d_prob, int nprob, int maxm, int p, int nb, int lo, int hi, int* err,
                  cudaStream_t st);
// The off-diagonal update of a blocked triangular solve (k_getrs_update's contract).
void oz_getrs_update(const SolveProb<double2>* d_prob, int nprob, int maxm, int maxrhs, int p, int nb, int lower, int* err,
                     cudaStream_t st);
