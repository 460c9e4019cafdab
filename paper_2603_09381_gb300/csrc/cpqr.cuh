// Batched column-pivoted QR with fresh column norms and the interpolative
// decomposition built from it (paper Sec. 3: ID via CPQR, adaptive rank).
#pragma once
#include <cuda_runtime.h>
#include "pm_common.cuh"

enum { CPQR_FIND_RANK = 0, CPQR_EXTEND = 1 };

// Pivot and reflector of a matrix's next step (q < 0: none, the phase is over).
template <typename C>
struct CpqrPick {
  int q;
  int ev;                        // complex128: shift of the pivot column's integers
  int reflect;                   // complex64: the pivot column is not zero
  C ctau, csc, sc, beta;         // conj(tau), conj(1 / (alpha - beta)), 1 / (alpha - beta) (complex128: scaled), R_ss
};

template <typename C>
struct CpqrProb {
  C* Z; int ld; int W; int n;    // W x n, factored in place (columns never move)
  double tol;
  int mode;                      // CPQR_FIND_RANK or CPQR_EXTEND
  int base;                      // steps already done when this phase starts
  int target;                    // stop before step `target`
  double* norm2;                 // 2 * n: squared trailing norms, ping-pong by step parity (-1: pivoted)
  int* perm;                     // perm[s] = column chosen at step s
  C* rdiag;                      // rdiag[s] = R_ss
  int* rank;                     // -1 until the rank criterion stops the factorization
  double* ref;                   // |R_11|
  CpqrPick<C>* pick;
  int* done;                     // chunks finished in the running step
  int* cexp;                     // complex128: column c holds integers of 2^(cexp[c] - 60)
  int* bad;                      // complex128: set to 1 if a column is not finite
};

struct CpqrChunk { int id; int c0; int c1; int first; };

template <typename C>
struct InterpProb {              // T (k x (n-k)) = R11^{-1} R12 in pivot order
  const C* Z; int ld; int n; int k;
  const int* perm; const C* rdiag;
  C* T; int ldt;
  C* R11;                        // k x k workspace (leading dimension k): R11 in pivot order
  const int* cexp;               // complex128: the columns' scales
};

template <typename C>
struct ScatterProb {             // dense L (rows = box positions) or R (columns = box positions)
  C* out; int ld; int off; int isL;
  const int* pos; const int* perm; int k; int ng;
  const C* T; int ldt;
};

template <typename S, typename D = S>
struct CopyProb { const S* src; int lds; D* dst; int ldd; int m; int n; };

struct PermFill { int* perm; int n; int done; };   // perm[done..n) <- unchosen columns, ascending

// Unpivoted blocked Householder QR of a tall Z (W x n, W > n) in place: the
// n x n triangle R ends in the top rows with zeros below its diagonal.  Column
// norms of every trailing block are those of Z, so the column-pivoted QR of R
// picks the pivots and R factor of Z's (exact arithmetic).
constexpr int QR_NB = 32;        // panel width
constexpr int QR_RB = 256;       // rows per block of the trailing update
template <typename C>
struct QrProb {
  C* Z; int ld; int W; int n;
  C* T;                          // QR_NB x QR_NB: compact-WY factor of the current panel
  C* V;                          // W x QR_NB (leading dimension W), or NULL: the panel's V
                                 // (rows j0.. at rows 0..) written out with its unit diagonal
  C* Yp;                         // update workspace: ceil(n/32) x mrb blocks of 32 x 32
  int mrb;                       // row blocks of QR_RB rows covering W
};
// Panels [j0, j0 + QR_NB) of every matrix with j0 < n; max_tiles = the most
// 32-column tiles right of a panel in any matrix.
// cluster: CTAs per matrix (1, 2, 4, 8), or 0 for as many as fill the SMs (the
// partial sums of a reflector, hence the last bits, depend on it).  max_w
// (complex128): the most rows of a matrix.
template <typename C>
void qr_panel(const QrProb<C>* d_prob, int nprob, int j0, cudaStream_t st, int cluster = 0, int max_w = 0);
// Trailing update of a complex128 panel (QR_NB reflectors, taus in T) on the
// tensor cores at FP64 accuracy: V holds QR_NB x (n - QR_NB) entries of Y, Yp
// ceil(n / 128) x mrb blocks of 128 x QR_NB partial sums, mrb = ceil(W / OZ_RB).
// *err is set if a bounded wait runs out.
constexpr int OZ_RB = 256;
void qr_update_oz(const QrProb<double2>* d_prob, int nprob, int j0, int max_n, int max_w, int* err, cudaStream_t st);
// max_rb: the most QR_RB-row blocks of rows j0..W-1 in any matrix.  With
// tc_err (complex64 only) the last step, C -= V Y, runs on the tensor cores
// (k_qr_apply_tc; max_w = the largest W), which set *tc_err if a bounded wait
// runs out; without it, on the CUDA cores.  no_arrive: see k_qr_apply_tc
// (tests of the timeout path).
template <typename C>
void qr_update(const QrProb<C>* d_prob, int nprob, int j0, int max_tiles, int max_rb, cudaStream_t st,
               int* tc_err = nullptr, int max_w = 0, bool no_arrive = false);
template <typename C>
void qr_zero_lower(const QrProb<C>* d_prob, int nprob, int max_n, cudaStream_t st);

void complete_perm(const PermFill* d_prob, int nprob, cudaStream_t st);
// Initial norms; complex128 columns go to fixed point (cexp) here, which has no
// NaN: *bad tells the host of columns that are not finite.
template <typename C>
void cpqr_init_norms(const CpqrProb<C>* d_prob, const CpqrChunk* d_chunk, int nchunk, cudaStream_t st);
// Before the first step of a phase (mode, base, target set): its first pivot.
template <typename C>
void cpqr_start(const CpqrProb<C>* d_prob, int nprob, cudaStream_t st);
// One elimination step (launch index t) of every active matrix; d_counter:
// a zeroed int, distinct for every launch (chunk dispenser).  tall: some
// complex64 matrix has W >= 2048 rows (selects the kernel instance with the
// register-resident column path).
template <typename C>
void cpqr_step(const CpqrProb<C>* d_prob, const CpqrChunk* d_chunk, int nchunk, int t, int* d_counter,
               cudaStream_t st, bool tall);
// The whole phase of the `count` matrices listed in d_list (h_n, h_w: their
// columns and rows), each in the shared memory of a cluster of at least cs
// CTAs (more while all of them fit on `sms` SMs); cpqr_resident_ctas: the fewest CTAs that hold an n-column, W-row
// matrix, or 0.  Norms as cpqr_init_norms leaves them; no cpqr_start needed.
template <typename C>
int cpqr_resident_ctas(int n, int W);
template <typename C>
void cpqr_resident(const CpqrProb<C>* d_prob, const int* d_list, const int* h_n, const int* h_w, int count, int cs,
                   int sms, cudaStream_t st);
// R11 (upper triangular, diagonal from rdiag) and R12 of every problem gathered
// in pivot order into R11 and T (ldt = k), for a blocked triangular solve
// T <- R11^{-1} T; max_elems = the largest k * n.
template <typename C>
void interp_gather(const InterpProb<C>* d_prob, int nprob, size_t max_elems, cudaStream_t st);
template <typename C>
void scatter_interp(const ScatterProb<C>* d_prob, int nprob, int max_elems, cudaStream_t st);
template <typename S, typename D>
void copy_batched(const CopyProb<S, D>* d_prob, int nprob, int max_elems, cudaStream_t st);

constexpr int CPQR_CB = 16;      // columns per chunk
