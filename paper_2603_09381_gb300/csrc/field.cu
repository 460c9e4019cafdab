// Off-boundary fields from a boundary solution (see field.cuh).  One CTA per
// evaluation point or direction sums the trapezoid rule over every node in a
// fixed order (block-wide reduction), so results are reproducible.  The near
// field's Hankel pair and the far field's sincos, which bound these kernels on
// the FP64 pipe together with 8 (far: 6) fused multiply-adds a right-hand side,
// are formed once for up to NR right-hand sides: 8 x 8 stars, 4,096 points and
// 720 directions, 8 right-hand sides: 65 ms with one CTA per right-hand side,
// 7.8 ms now.  Every fused operation is written out: left to the compiler, a
// right-hand side took 12 and its last bits depended on NR (10.1 ms).
#include "field.cuh"
#include "hankel.cuh"
#include "prof.cuh"
#include <type_traits>

namespace {

constexpr int FT = 256;

__device__ __forceinline__ double2 block_sum2(double2 v, double2* sh) {
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double2 t = make_double2(0, 0);
  if (threadIdx.x == 0)
    for (int w = 0; w < FT / 32; ++w) { t.x += sh[w].x; t.y += sh[w].y; }
  return t;
}

// q and u of node i: phi[row_off + l] and phi[row_off + n + l], l = i - node_off
__device__ __forceinline__ void qu_of(const InclDev* inc, const int* incl, const double2* phi, int i, double2& q,
                                      double2& u) {
  const InclDev d = inc[incl[i]];
  const int l = i - d.node_off;
  q = phi[d.row_off + l];
  u = phi[d.row_off + d.n + l];
}

// A thread's sums restart every RUN nodes and join its totals in shared memory:
// an FMA into the running sum rounds at the sum's size, several times a node
// (16,384 nodes, far field: rms error 3.33e-17 straight into the running sums,
// 2.99e-17 with each node's finished term added, 2.13e-17 with runs of 8, which take
// 2% of the case above).  With one run a thread (LONG false, up to RUN * FT nodes)
// the run is the total: the same bits without the totals, whose registers leave
// three CTAs an SM for four (1,720 nodes, 6 right-hand sides, 600 points and 232
// directions: 864 us with totals, 811 without).
constexpr int RUN = 8;
template <int NR, bool LONG>
struct RunSums {
  double2 acc[NR];
  double2 (*tot)[FT];
  int nodes = 0;
  __device__ __forceinline__ explicit RunSums(double2 (*t)[FT]) : tot(t) {
#pragma unroll
    for (int c = 0; c < NR; ++c) {
      acc[c] = make_double2(0, 0);
      if constexpr (LONG) tot[c][threadIdx.x] = make_double2(0, 0);
    }
  }
  __device__ __forceinline__ void flush() {
    if constexpr (LONG) {
#pragma unroll
      for (int c = 0; c < NR; ++c) {
        double2 t = tot[c][threadIdx.x];
        t.x += acc[c].x;
        t.y += acc[c].y;
        tot[c][threadIdx.x] = t;
        acc[c] = make_double2(0, 0);
      }
    }
  }
  __device__ __forceinline__ void next() {
    if constexpr (LONG)
      if ((++nodes & (RUN - 1)) == 0) flush();
  }
  __device__ __forceinline__ double2 total(int c) const {   // (after the last flush)
    if constexpr (LONG) return tot[c][threadIdx.x];
    else return acc[c];
  }
};

template <int NR, bool LONG>
__global__ void __launch_bounds__(FT) k_far_field(const InclDev* __restrict__ inc, NodesDev nd, int total, double k,
                                                  const double2* __restrict__ phi, int ldphi,
                                                  const double* __restrict__ ang, int ndir, double2* out) {
  __shared__ double2 sh[FT / 32], tot[LONG ? NR : 1][FT];
  const int dir = blockIdx.x;
  double sa, ca;
  sincos(ang[dir], &sa, &ca);
  RunSums<NR, LONG> sum(tot);
  for (int i = threadIdx.x; i < total; i += FT) {
    double s, co;
    sincos(-k * fma(ca, nd.x[i], sa * nd.y[i]), &s, &co);     // e^{-i k xhat.y}
    const double kn = k * fma(ca, nd.nx[i], sa * nd.ny[i]);
    const double w = nd.w[i];
    s *= w;
    co *= w;
#pragma unroll
    for (int c = 0; c < NR; ++c) {
      double2 q, u;
      qu_of(inc, nd.incl, phi + (size_t)c * ldphi, i, q, u);
      // -i k (xhat.n) u - q  (eps+ = 1)
      const double tx = fma(kn, u.y, -q.x), ty = fma(-kn, u.x, -q.y);
      double2& a = sum.acc[c];
      a.x = fma(-s, ty, fma(co, tx, a.x));
      a.y = fma(s, tx, fma(co, ty, a.y));
    }
    sum.next();
  }
  sum.flush();
#pragma unroll
  for (int c = 0; c < NR; ++c) {
    const double2 t = block_sum2(sum.total(c), sh);
    if (threadIdx.x == 0) {
      // gamma = (i/4) sqrt(2/(pi k)) e^{-i pi/4} = (sqrt(2/(pi k)) / 4) e^{i pi/4}
      const double gm = 0.25 * sqrt(2.0 / (3.141592653589793 * k)) * 0.7071067811865476;
      out[dir + (size_t)c * ndir] = make_double2(gm * (t.x - t.y), gm * (t.x + t.y));
    }
    __syncthreads();
  }
}

template <int NR, bool LONG>
__global__ void __launch_bounds__(FT) k_scattered(const InclDev* __restrict__ inc, NodesDev nd, int total, double k,
                                                  const double2* __restrict__ phi, int ldphi,
                                                  const double* __restrict__ xy, int npts, double2* out) {
  __shared__ double2 sh[FT / 32], tot[LONG ? NR : 1][FT];
  const int p = blockIdx.x;
  const double px = xy[2 * p], py = xy[2 * p + 1];
  RunSums<NR, LONG> sum(tot);
  for (int i = threadIdx.x; i < total; i += FT) {
    const double dx = px - nd.x[i], dy = py - nd.y[i];
    double r, ir, J0, Y0, J1, Y1;
    hk_distance(fma(dx, dx, dy * dy), r, ir);
    hankel01(k * r, J0, Y0, J1, Y1);
    const double w = 0.25 * nd.w[i], b = k * w * (fma(nd.nx[i], dx, nd.ny[i] * dy) * ir);
    // G = (i/4) H0 = (-Y0 + i J0)/4;  dG/dn_y = (i k/4) H1 b = k b (-Y1 + i J1)/4
    const double gx = -w * Y0, gy = w * J0, ex = -b * Y1, ey = b * J1;
#pragma unroll
    for (int c = 0; c < NR; ++c) {
      double2 q, u;
      qu_of(inc, nd.incl, phi + (size_t)c * ldphi, i, q, u);
      double2& a = sum.acc[c];
      a.x = fma(gy, q.y, fma(-gx, q.x, fma(-ey, u.y, fma(ex, u.x, a.x))));
      a.y = fma(-gy, q.x, fma(-gx, q.y, fma(ey, u.x, fma(ex, u.y, a.y))));
    }
    sum.next();
  }
  sum.flush();
#pragma unroll
  for (int c = 0; c < NR; ++c) {
    const double2 t = block_sum2(sum.total(c), sh);
    if (threadIdx.x == 0) out[p + (size_t)c * npts] = t;
    __syncthreads();
  }
}

// f(first right-hand side, group size as a constant, LONG as a constant) over
// groups of 8, 4, 2, 1
template <class F>
void rhs_groups(int nrhs, int total, F f) {
  for (int c = 0; c < nrhs;) {
    const int left = nrhs - c;
    const auto with = [&](auto nr) {
      if (total > RUN * FT) f(c, nr, std::true_type());
      else f(c, nr, std::false_type());
      c += nr;
    };
    if (left >= 8) with(std::integral_constant<int, 8>());
    else if (left >= 4) with(std::integral_constant<int, 4>());
    else if (left >= 2) with(std::integral_constant<int, 2>());
    else with(std::integral_constant<int, 1>());
    pm_launch_count_add(1);
  }
}

}  // namespace

void far_field(const InclDev* d_inc, NodesDev nodes, int total, double k0, const double2* phi, int ldphi, int nrhs,
               const double* d_angles, int ndir, double2* out, cudaStream_t st) {
  if (ndir <= 0 || nrhs <= 0) return;
  rhs_groups(nrhs, total, [&](int c, auto nr, auto runs) {
    k_far_field<decltype(nr)::value, decltype(runs)::value><<<ndir, FT, 0, st>>>(
        d_inc, nodes, total, k0, phi + (size_t)c * ldphi, ldphi, d_angles, ndir, out + (size_t)c * ndir);
  });
}

void scattered_field(const InclDev* d_inc, NodesDev nodes, int total, double k0, const double2* phi, int ldphi,
                     int nrhs, const double* d_xy, int npts, double2* out, cudaStream_t st) {
  if (npts <= 0 || nrhs <= 0) return;
  rhs_groups(nrhs, total, [&](int c, auto nr, auto runs) {
    k_scattered<decltype(nr)::value, decltype(runs)::value><<<npts, FT, 0, st>>>(
        d_inc, nodes, total, k0, phi + (size_t)c * ldphi, ldphi, d_xy, npts, out + (size_t)c * npts);
  });
}
