// Y = A X with the dense split operator (hi and lo planes, up to 8 columns of
// X) on the tensor cores, accurate to FP64: the residual products of the
// refinement.  The float-float products this replaces issued 12 FP32
// operations per real multiply-add (58 ms at N = 65,536, 70 ms with their sums
// folded into FP64); here an entry costs its cut into digits once, for all
// columns of X.  The cut's integer instructions bound the kernel (ALU pipe 69% busy;
// 28 ms at N = 65,536, 24 ms since hi and lo are cut together and two digits share
// a permutation); the read of the operator would take 10 ms.
//
// Digits as in oz.cuh, seven per number: relative to the largest part of its
// row within a fold of 128 or 512 columns (of X: of its column), each real is a
// 54-bit integer (both parts of an entry cut off).  What is left out (i + j > 6) is
// below 2^-49 of the product of the two maxima per real term.  Seven accumulators, one per digit i of A, take A_i times
// the digits 0 .. 6-i of X side by side (16 (7 - i) columns of TMEM each, 448 in
// all), so A_i is read once; a fold's sums stay below 2^24 and are exact.  At
// the end of a fold they are joined in integers and added in FP64.
//
// Graded columns.  Digits relative to the largest part of a row and of X's
// column lose what the row's large entries and X's large entries do not share:
// columns of small inclusions hold large entries and meet small ones of X.
// Where the columns' scales differ enough (colexp), A's columns are taken times
// 2^colexp and X's entries by as much less, on the exponents alone: nine stars,
// every other one 0.02 (0.03) of the others' size, 90 nodes: the refinement
// stalled at 3e-11 (2e-11) and reaches 2e-12 (7e-12) now, as it does with the
// FP64 product.  N = 65,536: 23.8 ms a product without, 24.8 with.
//
// One CTA of 17 warps per SM.  Two groups of 8 warps take alternate stages of
// 16 columns: load the planes (a stage ahead), cut the digits, store them to
// one of three buffers; one thread of the last warp issues the MMAs as buffers
// fill up.  All waits are bounded; one that runs out sets *err.
#include "operator.cuh"
#include "oz.cuh"
#include "oz_gemm.cuh"
#include "prof.cuh"
#include <algorithm>

namespace {

constexpr int NS = 7, TM = 128, KC = 16, KR = 2 * KC, BN = 16;
constexpr uint32_t SBO = (KR / 8) * 128;            // next 8 rows of an operand
constexpr uint32_t A_DIG = TM * KR * 2, B_DIG = BN * KR * 2;
constexpr uint32_t STAGE = NS * (A_DIG + B_DIG);
constexpr int NBUF = 3;
constexpr uint32_t OFF_BAR = NBUF * STAGE;          // full, empty, fold done, fold drained
constexpr int SMEM = OFF_BAR + 128;
constexpr int WORKERS = 512, T = WORKERS + 32;
constexpr int XCHUNK = NS * B_DIG / 16;             // uint4 of X's digits per stage
constexpr int WAIT = 1 << 20;

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(tcx::LBO >> 4) << 16 | (uint64_t)(SBO >> 4) << 32 |
         (uint64_t)1 << 46;
}
__device__ __forceinline__ uint32_t acc_col(int i) { return 16u * (7 * i - i * (i - 1) / 2); }
__device__ __forceinline__ uint32_t off(int row, int k) {
  return (uint32_t)(row >> 3) * SBO + (uint32_t)(k >> 3) * tcx::LBO + (uint32_t)(row & 7) * 16 + (uint32_t)(k & 7) * 2;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tcx::smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tcx::smem_u32(bar)) : "memory");
}

constexpr uint64_t BIAS = 0x0080808080808080ull;    // turns the seven digits into unsigned bytes

// hi + lo (lo of hi's sign and below hi's last place: SplitOp) relative to the
// exponent E as a 54-bit integer, each part cut off, plus BIAS.
__device__ __forceinline__ uint64_t cut(float hi, float lo, int E) {
  const uint32_t H = __float_as_uint(hi), L = __float_as_uint(lo);
  const int eh = (int)(H >> 23) & 0xFF, el = (int)(L >> 23) & 0xFF;
  const uint32_t mh = eh ? H << 8 | 0x80000000u : 0, ml = el ? L << 8 | 0x80000000u : 0;
  uint64_t q;
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"((uint64_t)mh << 32), "r"(E - eh + 10));   // (shifts past the width give 0)
  q += __funnelshift_rc(ml, 0u, (uint32_t)(E - el - 22));
  const int sg = (int)H >> 31;
  return (q ^ (uint64_t)(int64_t)sg) + BIAS + (uint32_t)(sg & 1);
}

// Digits I and I + 1 (I odd; 0: the largest) of two numbers as pairs of fp16
// (oz::digit_pairs), and digit 0 of two.
template <int I>
__device__ __forceinline__ uint2 digit_pairs(uint64_t a, uint64_t b) {
  constexpr int byte = 6 - I;
  const uint32_t x = byte >= 4 ? (uint32_t)(a >> 32) : (uint32_t)a, y = byte >= 4 ? (uint32_t)(b >> 32) : (uint32_t)b;
  constexpr uint32_t hi = (uint32_t)(byte & 3), sel = hi | (4 + hi) << 4 | (hi - 1) << 8 | (3 + hi) << 12;
  const uint32_t t = __byte_perm(x, y, sel);
  uint2 r = make_uint2(__byte_perm(t, 0x64646464u, 0x4140), __byte_perm(t, 0x64646464u, 0x4342));   // 1024 + byte
  asm("sub.f16x2 %0, %0, %1;" : "+r"(r.x) : "r"(0x64806480u));   // - 1152
  asm("sub.f16x2 %0, %0, %1;" : "+r"(r.y) : "r"(0x64806480u));
  return r;
}
__device__ __forceinline__ uint32_t digit0_pair(uint64_t a, uint64_t b) {
  uint32_t r = __byte_perm(__byte_perm((uint32_t)(a >> 32), (uint32_t)(b >> 32), 0x0062), 0x64646464u, 0x4140);
  asm("sub.f16x2 %0, %0, %1;" : "+r"(r) : "r"(0x64806480u));
  return r;
}
template <int I>
__device__ __forceinline__ void put2(unsigned char* p, const uint64_t* q) {
  const uint2 a = digit_pairs<I>(q[0], q[1]), b = digit_pairs<I>(q[2], q[3]), c = digit_pairs<I>(q[4], q[5]),
              d = digit_pairs<I>(q[6], q[7]);
  *reinterpret_cast<uint4*>(p + I * A_DIG) = make_uint4(a.x, b.x, c.x, d.x);
  *reinterpret_cast<uint4*>(p + (I + 1) * A_DIG) = make_uint4(a.y, b.y, c.y, d.y);
}
__device__ __forceinline__ void put8(unsigned char* p, const uint64_t* q) {
  *reinterpret_cast<uint4*>(p) = make_uint4(digit0_pair(q[0], q[1]), digit0_pair(q[2], q[3]), digit0_pair(q[4], q[5]),
                                            digit0_pair(q[6], q[7]));
  put2<1>(p, q);
  put2<3>(p, q);
  put2<5>(p, q);
}

constexpr int X_NOT_FINITE = 0xFFFF;

// Exponent of the largest part of X's column q in every 128 columns of A (a warp
// each), each entry's less its column's (colexp, or all zero).
__global__ void __launch_bounds__(256) k_x_exponents(const double2* __restrict__ X, int ldx, int N, int nrhs,
                                                     const signed char* __restrict__ colexp,
                                                     unsigned short* __restrict__ xexp) {
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int c = w >> 3, q = w & 7;
  if (c * 128 >= N) return;
  int e = 0;
  if (q < nrhs)
    for (int k = c * 128 + lane; k < min(N, c * 128 + 128); k += 32) {
      const double2 v = X[k + (size_t)q * ldx];
      const int x = max(oz::exponent(v.x), oz::exponent(v.y));
      e = max(e, x == 0x7FF ? X_NOT_FINITE : x - (colexp ? colexp[k] : 0));
    }
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) xexp[c * 8 + q] = (unsigned short)e;
}

// X's digits in the stages' layout: rows 0 .. 7 (real outputs) hold [xr | -xi],
// rows 8 .. 15 (imaginary outputs) [xi | xr].  A CTA per stage, a thread per
// (column, k).
__global__ void __launch_bounds__(128) k_x_digits(const double2* __restrict__ X, int ldx, int N, int nrhs, int fold,
                                                  const signed char* __restrict__ colexp,
                                                  const unsigned short* __restrict__ xexp, unsigned char* __restrict__ out) {
  const int t = blockIdx.x, q = threadIdx.x >> 4, kk = threadIdx.x & 15, k = t * KC + kk;
  const int c0 = t * KC / (128 * fold) * fold;
  int E = 0;
  for (int c = c0; c < c0 + fold && c * 128 < N; ++c) E = max(E, (int)xexp[c * 8 + q]);
  if (colexp && k < N) E += colexp[k];
  const double2 v = k < N && q < nrhs ? X[k + (size_t)q * ldx] : make_double2(0.0, 0.0);
  // 54 bits: oz::digits' 62 less the lowest byte
  auto cut_x = [&](double x, bool neg) { return (uint64_t)((int64_t)(oz::digits(x, E, neg) - oz::BIAS + 128) >> 8) + BIAS; };
  const uint64_t r = cut_x(v.x, false), i = cut_x(v.y, false), ni = cut_x(v.y, true);
  unsigned char* o = out + (size_t)t * (NS * B_DIG);
  auto put = [&](uint64_t a, int row, int col) {
    const uint2 d1 = digit_pairs<1>(a, 0), d3 = digit_pairs<3>(a, 0), d5 = digit_pairs<5>(a, 0);
    const uint32_t d[NS] = {digit0_pair(a, 0), d1.x, d1.y, d3.x, d3.y, d5.x, d5.y};
#pragma unroll
    for (int s = 0; s < NS; ++s) *reinterpret_cast<unsigned short*>(o + s * B_DIG + off(row, col)) = (unsigned short)d[s];
  };
  put(r, q, kk);
  put(ni, q, KC + kk);
  put(i, 8 + q, kk);
  put(r, 8 + q, KC + kk);
}

// Exponent of the largest part of every row in every 128 columns (where the
// FP32 product, which records them as it goes, has not run, or with colexp,
// which it does not know), each entry's plus its column's.
__global__ void __launch_bounds__(128) k_row_exponents(const float2* __restrict__ Ah, size_t lda, int N,
                                                       const signed char* __restrict__ colexp,
                                                       unsigned char* __restrict__ rexp) {
  const int row = blockIdx.x * 128 + threadIdx.x, c = blockIdx.y;
  if (row >= N) return;
  int e = 0;
#pragma unroll 8
  for (int k = c * 128; k < min(N, c * 128 + 128); ++k) {
    const float2 v = __ldg(Ah + row + (size_t)k * lda);
    const int x = (int)(max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu) >> 23);
    e = max(e, x == 0xFF ? x : x + (colexp ? colexp[k] : 0));
  }
  rexp[row + (size_t)c * N] = (unsigned char)e;
}

// GRADED: with colexp.  Rows [128 blockIdx.x, + 128), folds [blockIdx.y * folds, + folds) of 128 * fold columns.
template <bool GRADED>
__global__ void __launch_bounds__(T, 1) k_dense_matvec_oz(const float2* __restrict__ Ah, const float2* __restrict__ Al,
                                                          size_t lda, int N, const unsigned char* __restrict__ rexp,
                                                          const signed char* __restrict__ colexp,
                                                          const unsigned short* __restrict__ xexp,
                                                          const uint4* __restrict__ Xd, double2* __restrict__ Y, int ldy,
                                                          int nrhs, int fold, int folds, int* err, int no_arrive) {
  extern __shared__ __align__(1024) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + OFF_BAR);
  uint64_t* empty = full + NBUF;
  uint64_t* done = empty + NBUF;      // a fold's MMAs have finished
  uint64_t* drained = done + 1;       // its accumulators have been read
  uint64_t* last = drained + 1;       // nothing is in flight any more
  uint64_t* never = last + 1;         // tests of the timeout path: nothing arrives at it
  uint32_t* taddr = reinterpret_cast<uint32_t*>(never + 1);
  int* s_fail = reinterpret_cast<int*>(taddr + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < NBUF; ++i) { mbar_init(&full[i], 256); mbar_init(&empty[i], 1); }
    mbar_init(done, 1);
    mbar_init(last, 1);
    mbar_init(never, 1);
    mbar_init(drained, WORKERS);
    *s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tcx::smem_u32(taddr)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *taddr;
  if (no_arrive) {   // see oz::begin
    if (!tcx::mbar_wait(never, 0, 1 << 10)) *(volatile int*)s_fail = 1;
    __syncthreads();
  }
  const int spf = 8 * fold;                                  // stages per fold
  const int t0 = (int)blockIdx.y * folds * spf, t1 = min((N + KC - 1) / KC, t0 + folds * spf);
  const int row0 = blockIdx.x * TM;
  // a wait that ran out anywhere ends all waiting; nothing is issued or written after it
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (*(volatile int*)s_fail) return;
    if (!tcx::mbar_wait(bar, parity, WAIT)) *(volatile int*)s_fail = 1;
  };
  if (warp == WORKERS / 32) {
    if (lane == 0) {
      for (int t = t0; t < t1; ++t) {
        const int n = t - t0, b = n % NBUF;
        if (n % spf == 0 && n > 0) wait(drained, (uint32_t)((n / spf - 1) & 1));
        wait(&full[b], (uint32_t)((n / NBUF) & 1));
        if (*(volatile int*)s_fail) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t as = tcx::smem_u32(sm) + b * STAGE, bs = as + NS * A_DIG;
#pragma unroll
        for (int ks = 0; ks < KR / 16; ++ks)
#pragma unroll
          for (int i = 0; i < NS; ++i)
            oz::mma(tmem + acc_col(i), sdesc(as + i * A_DIG + ks * 2 * tcx::LBO), sdesc(bs + ks * 2 * tcx::LBO),
                    oz::idesc(BN * (NS - i)), n % spf > 0 || ks > 0 ? 1u : 0u);
        tcx::mma_commit(&empty[b]);
        if (n % spf == spf - 1 || t == t1 - 1) tcx::mma_commit(done);
      }
      tcx::mma_commit(last);   // also after a wait that ran out: TMEM is freed below
      if (!tcx::mbar_wait(last, 0, WAIT)) *(volatile int*)s_fail = 1;
    }
    __syncwarp();
  } else {
    const int g = warp >> 3, u = tid & 255, r = u & 127, kg = u >> 7, row = row0 + r;
    const int orow = row0 + 32 * (warp & 3) + lane, cg = 4 * (warp >> 2);   // outputs: row, real columns cg .. cg + 3
    float2 h[8], l[8];
    uint4 x0 = make_uint4(0, 0, 0, 0), x1 = x0;
    uint2 ce = make_uint2(0, 0);   // GRADED: the eight columns' exponents, a byte each
    auto load = [&](int t) {
      const int k = t * KC + 8 * kg;
      if (GRADED) ce = __ldg(reinterpret_cast<const uint2*>(colexp + k));   // (padded to a multiple of 128 columns)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const bool in = row < N && k + i < N;
        h[i] = in ? __ldg(Ah + row + (size_t)(k + i) * lda) : make_float2(0.f, 0.f);
        l[i] = in ? __ldg(Al + row + (size_t)(k + i) * lda) : make_float2(0.f, 0.f);
      }
      if (u < XCHUNK / 2) {
        x0 = __ldg(Xd + (size_t)t * XCHUNK + u);
        x1 = __ldg(Xd + (size_t)t * XCHUNK + XCHUNK / 2 + u);
      }
    };
    auto row_exp = [&](int rr, int f) {
      int e = 1;
      for (int c = f * fold; c < (f + 1) * fold && c * 128 < N; ++c) if (rr < N) e = max(e, (int)rexp[rr + (size_t)c * N]);
      return e;
    };
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (t0 + g < t1) load(t0 + g);
    int f = t0 / spf, E = row_exp(row, f);
    for (int f0 = t0; f0 < t1; f0 += spf, ++f) {
      const int fend = min(t1, f0 + spf);
      for (int t = f0 + g; t < fend; t += 2) {   // spf is even: a group keeps its parity
        const int n = t - t0, b = n % NBUF;
        if (n >= NBUF) wait(&empty[b], (uint32_t)((n / NBUF - 1) & 1));
        unsigned char* A = sm + b * STAGE;
        uint64_t q[8];
        auto e_of = [&](int i) {
          return GRADED ? E - (int)(signed char)((i < 4 ? ce.x : ce.y) >> (8 * (i & 3))) : E;
        };
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = cut(h[i].x, l[i].x, e_of(i));
        put8(A + off(r, 8 * kg), q);
#pragma unroll
        for (int i = 0; i < 8; ++i) q[i] = cut(h[i].y, l[i].y, e_of(i));
        put8(A + off(r, KC + 8 * kg), q);
        if (u < XCHUNK / 2) {
          uint4* B = reinterpret_cast<uint4*>(A + NS * A_DIG);
          B[u] = x0;
          B[XCHUNK / 2 + u] = x1;
        }
        if (t + 2 < t1) load(t + 2);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(&full[b]);
      }
      // the fold's sums: S_s = sum over i of accumulator i's digit s - i
      wait(done, (uint32_t)(((f0 - t0) / spf) & 1));
      asm volatile("tcgen05.fence::after_thread_sync;");
      if (__all_sync(0xffffffffu, *(volatile int*)s_fail == 0)) {
        const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cg;
        int64_t hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
#pragma unroll
        for (int s = 0; s < NS; ++s) {
          float v[NS][4];
#pragma unroll
          for (int i = 0; i <= s; ++i) oz::tmem_ld4(base + acc_col(i) + 16 * (s - i), v[i]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            int sum = 0;
#pragma unroll
            for (int i = 0; i <= s; ++i) sum += __float2int_rn(v[i][j]);
            // V = sum_s S_s 2^(8 (6 - s)) = hi 2^32 + lo
            if (s <= 2) hi[j] += (int64_t)sum << (8 * (2 - s)); else lo[j] += (int64_t)sum << (8 * (6 - s));
          }
        }
        const int eo = row_exp(orow, f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          int ex = 0;
          for (int c = f * fold; c < (f + 1) * fold && c * 128 < N; ++c) ex = max(ex, (int)xexp[c * 8 + ((cg + j) & 7)]);
          const double d = oz::join(hi[j], lo[j], eo + ex - 1208);
          acc[j] += eo == 0xFF || ex == X_NOT_FINITE ? __longlong_as_double(0x7FF8000000000000ll) : d;
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      mbar_arrive(drained);
      if (fend < t1) E = row_exp(row, f + 1);
    }
    if (orow < N && *(volatile int*)s_fail == 0) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = cg + j, qq = c & 7;
        if (qq < nrhs) {
          double* y = reinterpret_cast<double*>(Y + orow + (size_t)qq * ldy) + (c >> 3);
          atomicAdd(y, acc[j]);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  if (tid == 0 && *(volatile int*)s_fail) atomicExch(err, 1);
}

}  // namespace

void dense_row_exponents(SplitOp A, int N, const signed char* colexp, unsigned char* rexp, cudaStream_t st) {
  if (N <= 0) return;
  k_row_exponents<<<dim3((N + 127) / 128, (N + 127) / 128), 128, 0, st>>>(A.hi, A.ld, N, colexp, rexp);
  pm_launch_count_add(1);
}

size_t dense_matvec_oz_bytes(int N) { return (size_t)((N + 127) / 128) * 128 / KC * (NS * B_DIG); }

void dense_matvec_oz(SplitOp A, int N, const unsigned char* rexp, const signed char* colexp, const double2* X, int ldx,
                     double2* Y, int ldy, int nrhs, unsigned char* xdig, unsigned short* xexp, int* err,
                     cudaStream_t st) {
  if (N <= 0 || nrhs <= 0) return;
  for (int q = 0; q < nrhs; ++q) cudaMemsetAsync(Y + (size_t)q * ldy, 0, sizeof(double2) * N, st);
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // the same value every time: idempotent across threads and devices
  const auto kernel = colexp ? k_dense_matvec_oz<true> : k_dense_matvec_oz<false>;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  const int rb = (N + TM - 1) / TM, chunks = (N + 127) / 128;
  // long folds cost the least; short ones let a small matrix use more SMs
  const int fold = (long)rb * ((chunks + 3) / 4) >= 2 * sms ? 4 : 1;
  const int nf = (chunks + fold - 1) / fold;
  // about four waves of CTAs, the column range of each a whole number of folds
  const int segs = std::max(1, std::min(nf, (4 * sms + rb - 1) / rb)), folds = (nf + segs - 1) / segs;
  KPROF_BEGIN(st);
  for (int r0 = 0; r0 < nrhs; r0 += 8) {
    const int nr = std::min(8, nrhs - r0);
    k_x_exponents<<<chunks, 256, 0, st>>>(X + (size_t)r0 * ldx, ldx, N, nr, colexp, xexp);
    k_x_digits<<<(N + KC - 1) / KC, 128, 0, st>>>(X + (size_t)r0 * ldx, ldx, N, nr, fold, colexp, xexp, xdig);
    kernel<<<dim3(rb, (nf + folds - 1) / folds), T, SMEM, st>>>(
        A.hi, A.lo, A.ld, N, rexp, colexp, xexp, (const uint4*)xdig, Y + (size_t)r0 * ldy, ldy, nr, fold, folds, err,
        g_oz_no_arrive);
    pm_launch_count_add(3);
  }
  KPROF_END(st, "dense_matvec_oz", 0.0);
}
