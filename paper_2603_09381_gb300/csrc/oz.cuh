// Complex128 products on the tensor cores, accurate to FP64 (the Ozaki
// scheme: K. Ozaki, T. Ogita, S. Oishi, S. Rump, "Error-free transformations
// of matrix multiplication by using fast routines of matrix multiplication",
// Numer. Algorithms 59 (2012), with integer digits held in fp16).
//
// Why: GB300's FP64 pipe does 2 fused multiply-adds per clock and SM
// (1.26 TFLOP/s measured for the chip), its tensor cores 4096 in fp16.  An
// FP64 product as 36 exact fp16 products leaves the FP64 pipe one addition
// per output and stage of 32 complex terms instead of 128 fused
// multiply-adds.
//
// A stage multiplies a 128 x 32 by a 32 x 32 complex block.  Every row of A
// and every column of B has, per stage, the exponent of its largest part;
// relative to it each real is rounded to a 62-bit integer (nine bits more
// than a double holds, for rows and columns of graded entries) and cut into
// eight balanced base-256 digits, exact in fp16.  The products of digits i
// and j of equal i + j = s <= 7 add up in one FP32 accumulator: at most
// 64 x 8 products of at most 2^14, 2^23, hence exact.  What is left out
// (s > 7) is below 2^-57 of the product of the two maxima per real term: the
// error is relative to those, not to each term, so that a row and a column
// graded in opposite directions lose what their large parts do not share (the
// callers' matrices are kept from that by their unit of length, length_unit in
// runtime.cu).  The eight sums are
// joined in a 75-bit integer, rounded once to a double and added in FP64.  A
// stage's result depends only on its row of A and its column of B, so the
// tiling changes no bit.
//
// Layout: the real form [Ar | Ai] (128 x 64) times [[Br, Bi], [-Bi, Br]]
// (64 x 64: real columns, then imaginary), A's digits as eight 128 x 64
// operands, B's as eight 64 x 64 ones, one 64-column accumulator for each sum
// (all 512 TMEM columns).  All MMAs have one shape and each sum its own
// columns: MMAs of several widths on overlapping columns are not ordered among
// themselves.  K-major, no swizzle: the core matrices are written by
// conflict-free 16-byte stores.  195 KB of shared memory: one CTA per SM.
//
// What bounds a stage is that its phases (load, cut, MMAs, join) come one after
// the other on 16 warps an SM, behind barriers: ALU pipe 37-40% busy, FP64 15-23%,
// tensor 16-18%, 32% of the issue slots.  The integer instructions are its largest
// part: the join in 32-bit words and two digits to one permutation took 8 x 8 stars
// from 336 to 320 ms.
#pragma once
#include "pm_common.cuh"
#include "tc_common.cuh"

namespace oz {

constexpr int T = 512;          // threads: (row, group of 8 k) for A; TMEM lane and 8 columns in the epilogue
constexpr int TM = 128;         // complex rows of a tile
constexpr int TN = 32;          // complex columns of a tile
constexpr int TKC = 32;         // complex k of a stage
constexpr int NS = 8;           // digits
constexpr int KR = 2 * TKC;     // real k of a stage
constexpr uint32_t SBO = (KR / 8) * 128;             // next 8 rows of an operand
constexpr uint32_t A_BYTES = TM * KR * 2;            // one digit of A
constexpr uint32_t B_BYTES = 2 * TN * KR * 2;        // one digit of B
constexpr uint32_t OFF_B = NS * A_BYTES;
constexpr uint32_t OFF_EXP = OFF_B + NS * B_BYTES;   // per k group: exponents of A's rows, then B's columns; B's overall
constexpr uint32_t OFF_BAR = OFF_EXP + (4 * (TM + TN) + TN) * 4;
constexpr int SMEM = OFF_BAR + 32;
constexpr int WAIT = 1 << 20;   // x ~1 us suspend hint: about a second

// kind::f16 instruction descriptor: D f32 (bit 4), A and B fp16 (0), N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t idesc(int N) { return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TM >> 4) << 24); }
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(tcx::LBO >> 4) << 16 | (uint64_t)(SBO >> 4) << 32 |
         (uint64_t)1 << 46;
}
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t id, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          tmem),
      "l"(ad), "l"(bd), "r"(id), "r"(accumulate));
}
// four consecutive fp32 columns of this thread's TMEM lane, not waited for
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* d) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
               : "r"(taddr));
}

__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// x relative to the exponent E >= exponent(x) as a 62-bit integer, plus the
// bias that turns its base-256 digits into unsigned bytes; neg: of -x.
// Subnormal x counts as zero.
constexpr uint64_t BIAS = 0x8080808080808080ull;
__device__ __forceinline__ uint64_t digits(double x, int E, bool neg) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  const int e = (int)(h >> 20) & 0x7FF, d = e ? min(E - e, 63) : 63;   // 63 leaves nothing
  const uint64_t m = (uint64_t)((h & 0xFFFFFu) | 0x100000u) << 32 | (uint32_t)__double2loint(x);
  const uint64_t q = ((m << 10 >> d) + 1) >> 1;                        // rounded
  const int sg = ((int)h >> 31) ^ (neg ? -1 : 0);
  return (q ^ (uint64_t)(int64_t)sg) + BIAS + (uint32_t)(sg & 1);
}

// Digits I and I + 1 (I even; 0: the largest) of two numbers as pairs of fp16:
// bytes go through 1024 + byte (exact in fp16) to the signed digit.
template <int I>
__device__ __forceinline__ uint2 digit_pairs(uint64_t a, uint64_t b) {
  constexpr int byte = 7 - I;
  const uint32_t x = byte >= 4 ? (uint32_t)(a >> 32) : (uint32_t)a, y = byte >= 4 ? (uint32_t)(b >> 32) : (uint32_t)b;
  constexpr uint32_t hi = (uint32_t)(byte & 3), sel = hi | (4 + hi) << 4 | (hi - 1) << 8 | (3 + hi) << 12;
  const uint32_t t = __byte_perm(x, y, sel);             // a's and b's byte of digit I, then of I + 1
  uint2 r = make_uint2(__byte_perm(t, 0x64646464u, 0x4140), __byte_perm(t, 0x64646464u, 0x4342));   // 0x64 above each
  asm("sub.f16x2 %0, %0, %1;" : "+r"(r.x) : "r"(0x64806480u));   // - 1152
  asm("sub.f16x2 %0, %0, %1;" : "+r"(r.y) : "r"(0x64806480u));
  return r;
}
template <int I>
__device__ __forceinline__ void put2(unsigned char* p, uint32_t step, const uint64_t* q) {
  const uint2 a = digit_pairs<I>(q[0], q[1]), b = digit_pairs<I>(q[2], q[3]), c = digit_pairs<I>(q[4], q[5]),
              d = digit_pairs<I>(q[6], q[7]);
  *reinterpret_cast<uint4*>(p + I * step) = make_uint4(a.x, b.x, c.x, d.x);
  *reinterpret_cast<uint4*>(p + (I + 1) * step) = make_uint4(a.y, b.y, c.y, d.y);
}
// the eight digits of eight numbers into eight operands `step` bytes apart
__device__ __forceinline__ void put8(unsigned char* p, uint32_t step, const uint64_t* q) {
  put2<0>(p, step, q);
  put2<2>(p, step, q);
  put2<4>(p, step, q);
  put2<6>(p, step, q);
}
__device__ __forceinline__ uint32_t row_off(int row, int k) { return (uint32_t)(row >> 3) * SBO + (uint32_t)(k >> 3) * tcx::LBO + (uint32_t)(row & 7) * 16; }

// The double nearest to (hi 2^32 + lo) 2^p2, |hi| and |lo| below 2^62; in
// 32-bit words, as 64-bit shifts by a variable take three instructions each and
// a stage's epilogue is its largest part.
__device__ __forceinline__ double join(int64_t hi, int64_t lo, int p2) {
  hi += lo >> 32;                       // = hi 2^32 + l, 0 <= l < 2^32
  const uint32_t sg = (uint32_t)((int32_t)(hi >> 32) >> 31);
  uint32_t w2 = (uint32_t)(hi >> 32) ^ sg, w1 = (uint32_t)hi ^ sg, w0 = (uint32_t)lo ^ sg;   // magnitude
  asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, 0;\n addc.u32 %2, %2, 0;" : "+r"(w0), "+r"(w1), "+r"(w2) : "r"(sg & 1));
  int e = 1023 + 95 + p2;
  if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; e -= 32; }
  if (w2 == 0) { w2 = w1; w1 = w0; e -= 32; }
  const int lz = __clz((int)w2);
  const uint32_t m1 = __funnelshift_l(w1, w2, lz), m0 = __funnelshift_l(w0, w1, lz);
  e -= lz;
  uint64_t r = ((uint64_t)m1 << 32 | m0) >> 11;
  r += (m0 >> 10) & 1;                  // 53 bits (a carry goes on into the exponent)
  r += (uint64_t)((uint32_t)(e - 1) << 20 | (sg & 0x80000000u)) << 32;
  if (m1 == 0 || e <= 0) r = 0;
  if (e >= 2047) r = (uint64_t)(sg & 0x80000000u | 0x7FF00000u) << 32;
  return __longlong_as_double((long long)r);
}
// The double nearest to V 2^(ex - 2112), V = sum_s v_s 2^(8 (7 - s)); ex: the
// sum of the two exponents, or negative for a row or column that is not finite.
__device__ __forceinline__ double join(const float* v, int ex) {
  // |v_s| <= (s + 1) 2^20: pairs of sums fit 32 bits
  const int p0 = __float2int_rn(v[0]) * 256 + __float2int_rn(v[1]), p1 = __float2int_rn(v[2]) * 256 + __float2int_rn(v[3]);
  const int p2 = __float2int_rn(v[4]) * 256 + __float2int_rn(v[5]), p3 = __float2int_rn(v[6]) * 256 + __float2int_rn(v[7]);
  const double r = join((int64_t)p0 * 65536 + p1, (int64_t)p2 * 65536 + p3, ex - 2112);
  return ex < 0 ? __longlong_as_double(0x7FF8000000000000ll) : r;
}

struct Cta {
  unsigned char* sm;
  uint32_t tmem;
  uint32_t phase;
  bool ok;   // no wait has run out: the same in every thread of the CTA
};

// All threads of the CTA; smem: oz::SMEM bytes of dynamic shared memory, 128-byte aligned.
// no_arrive (tests of the timeout path): the CTA first waits, with a bound of
// about a millisecond, on a barrier that nothing arrives at.
__device__ __forceinline__ Cta begin(unsigned char* sm, int no_arrive) {
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + OFF_BAR);   // a stage's MMAs; then the drain's (end)
  uint32_t* taddr = reinterpret_cast<uint32_t*>(sm + OFF_BAR + 16);
  if (threadIdx.x == 0) {
    tcx::mbar_init(bar);
    tcx::mbar_init(bar + 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tcx::smem_u32(taddr)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  Cta c{sm, *taddr, 0, true};
  if (no_arrive) c.ok = __syncthreads_and(tcx::mbar_wait(bar + 1, 0, 1 << 10) ? 1 : 0) != 0;
  return c;
}
// After a wait that ran out nothing more was cut, issued or stored (stage); the
// MMAs still in flight are waited for, with a limit, at a barrier of their own
// (thread 0 issued them all), so that no earlier phase can stand in for theirs.
__device__ __forceinline__ void end(Cta& c, int* err) {
  if (!c.ok && threadIdx.x == 0) {
    uint64_t* drain = reinterpret_cast<uint64_t*>(c.sm + OFF_BAR) + 1;
    tcx::mma_commit(drain);
    tcx::mbar_wait(drain, 0, WAIT);
    atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(c.tmem), "r"(512));
}

// One stage: emit(j, part, d) receives the real (part 0) and imaginary parts
// of (A B)(row, 8 cg + j), j = 0 .. 7, for this thread's row (32 (warp % 4) +
// lane) and column group cg = warp / 4.  a(row, k) and b(k, col) return the
// operands' entries, zero outside; new_a: A's digits are not in shared memory
// yet; during() runs while the MMAs do (loads for emit).  All 512 threads call it.
template <class FA, class FB, class FE, class FD>
__device__ __forceinline__ void stage(Cta& c, bool new_a, const FA& a, const FB& b, const FE& emit, const FD& during) {
  if (!c.ok) return;   // a wait ran out before: the operands may still be read
  const int tid = threadIdx.x, warp = tid >> 5;
  int* ea = reinterpret_cast<int*>(c.sm + OFF_EXP);   // [k group][row]
  int* eb = ea + 4 * TM;                              // [k group][column]
  int* ebm = eb + 4 * TN;                             // [column]: the largest, far below zero if not finite
  const int row = tid & (TM - 1), kg = tid >> 7;
  const int bn = tid & 31, bg = (tid >> 5) & 3, bpart = tid >> 7;   // B: threads 0 .. 255
  double2 va[8];
  if (new_a) {
    int e = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) va[i] = a(row, 8 * kg + i);
#pragma unroll
    for (int i = 0; i < 8; ++i) e = max(e, max(exponent(va[i].x), exponent(va[i].y)));
    ea[kg * TM + row] = e;
  }
  double vb[8];
  if (tid < 256) {
    int e = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double2 v = b(8 * bg + i, bn);
      e = max(e, max(exponent(v.x), exponent(v.y)));
      vb[i] = bpart ? v.y : v.x;
    }
    if (bpart == 0) eb[bg * TN + bn] = e;
  }
  __syncthreads();
  if (new_a) {
    const int E = max(max(ea[row], ea[TM + row]), max(ea[2 * TM + row], ea[3 * TM + row]));
    uint64_t q[8];
    unsigned char* p = c.sm + row_off(row, 8 * kg);
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = digits(va[i].x, E, false);
    put8(p, A_BYTES, q);
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = digits(va[i].y, E, false);
    put8(p + (TKC / 8) * tcx::LBO, A_BYTES, q);
  }
  if (tid < 256) {
    const int E = max(max(eb[bn], eb[TN + bn]), max(eb[2 * TN + bn], eb[3 * TN + bn]));
    if (tid < TN) ebm[bn] = E == 0x7FF ? -0x4000 : E;
    // real part: [row bn, k] and [row 32 + bn, 32 + k]; imaginary part: negated [row bn, 32 + k], [row 32 + bn, k]
    uint64_t q[8];
    unsigned char* B = c.sm + OFF_B;
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = digits(vb[i], E, false);
    put8(B + row_off(TN + bn, (bpart ? 0 : TKC) + 8 * bg), B_BYTES, q);
    if (bpart) {
#pragma unroll
      for (int i = 0; i < 8; ++i) q[i] = 2 * BIAS - q[i];
    }
    put8(B + row_off(bn, (bpart ? TKC : 0) + 8 * bg), B_BYTES, q);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  uint64_t* bar = reinterpret_cast<uint64_t*>(c.sm + OFF_BAR);
  if (tid == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t as = tcx::smem_u32(c.sm), bs = as + OFF_B;
    for (int ks = 0; ks < KR / 16; ++ks) {
      const uint32_t ko = ks * 2 * tcx::LBO;   // 16 fp16 along k = two core matrices
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        const uint64_t ad = sdesc(as + i * A_BYTES + ko);
#pragma unroll
        for (int j = 0; j < NS - i; ++j)
          mma(c.tmem + (i + j) * 2 * TN, ad, sdesc(bs + j * B_BYTES + ko), idesc(2 * TN), ks + i > 0 ? 1u : 0u);
      }
    }
    tcx::mma_commit(bar);
  }
  // the exponents of this thread's outputs, while the MMAs run
  const int er = 32 * (warp & 3) + (tid & 31), cg = warp >> 2;
  int E = max(max(ea[er], ea[TM + er]), max(ea[2 * TM + er], ea[3 * TM + er]));
  if (E == 0x7FF) E = -0x4000;
  during();
  const bool done = tcx::mbar_wait(bar, c.phase, WAIT);
  c.phase ^= 1;
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (__all_sync(0xffffffffu, done ? 1 : 0)) {
    const uint32_t t0 = c.tmem + ((uint32_t)((warp & 3) * 32) << 16) + 8 * cg;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int4 F = *reinterpret_cast<const int4*>(ebm + 8 * cg + 4 * h);
      const int ef[4] = {E + F.x, E + F.y, E + F.z, E + F.w};
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        float v[NS][4];
#pragma unroll
        for (int s = 0; s < NS; ++s) tmem_ld4(t0 + s * 2 * TN + part * TN + 4 * h, v[s]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float w[NS] = {v[0][j], v[1][j], v[2][j], v[3][j], v[4][j], v[5][j], v[6][j], v[7][j]};
          const double d = join(w, ef[j]);
          emit(4 * h + j, part, d);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  c.ok = __syncthreads_and(done ? 1 : 0) != 0;   // the operands and accumulators may be overwritten
  asm volatile("tcgen05.fence::after_thread_sync;");
}

}  // namespace oz
