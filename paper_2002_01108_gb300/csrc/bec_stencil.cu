// All-at-once stencil kernels (Sec. 2, eq. allatoncesystem): L v, P_eps v,
// the right-hand side f and the true residual RES of Sec. 5.
//
// With M = I and K = (a/h^2) x (3- or 5-point Laplacian), block row n of L is
//     (L v)^n = (1 + 2 dim c) v^n - c (sum of the 2 dim neighbours of v^n) - v^{n-1},
// c = tau a / h^2, with no v^0 term; P_eps adds -eps v^N to block row 1.  With
// Q1 elements (Example 1 of Sec. 5) it is (M + tau K) v^n - M v^{n-1}, with the
// 9-point stencils of M and K, and P_eps adds -eps M v^N.  The two-step
// scheme (eq. pstepscheme with r = (3/2, -2, 1/2), template parameter P = 2)
// has block rows (r0 M + tau K) v^n + r1 M v^{n-1} + r2 M v^{n-2}, and P_eps
// wraps the missing terms around with the factor eps (eq.
// pstepbecpreconditioner).
// A thread owns one spatial point and walks a chunk of time slices, keeping
// v^{n-1} in a register, so v is read from memory once.
#include <cuda_runtime.h>

#include <cmath>

#include "bec_fx.cuh"
#include "bec_internal.h"

namespace bec {
namespace {

constexpr int kStencilThreads = 256;
constexpr int kTimeChunk = 8;

struct StencilGeom {
  long long J;
  int m, N, dim;
  double c;       // tau a / h^2 (constant a)
  double alpha;   // (1 + 2 dim c) / c
  const double* __restrict__ kc;   // variable a: tau K row [centre, W, E, S, N] x J, or null
  // Q1 elements (q1 != 0): the 9-point (2D) or 3-point (1D) stencils of
  // M + tau K and of M, as centre / edge / corner weights
  int q1;
  double ac, ae, ak, mc, me, mk;
  // two-step scheme: r1, r2 of the rows; rhs1, rhs2 = the multiples of M u^0
  // that the right-hand side adds to slices 1 and 2 (BDF1: 1 and 0)
  double r1, r2, rhs1, rhs2;
};

// sums of the 4 edge and 4 corner neighbours of point q of slice s (zero
// outside the interior; 1D: the 2 neighbours, no corners)
__device__ __forceinline__ void neighbour_sums(const double* __restrict__ s, long long q, int ix,
                                               int iy, const StencilGeom& g, double& edge,
                                               double& corner) {
  const int m = g.m;
  const bool w = ix > 0, e = ix < m - 1;
  edge = (w ? s[q - 1] : 0.0) + (e ? s[q + 1] : 0.0);
  corner = 0.0;
  if (g.dim == 2) {
    const bool so = iy > 0, no = iy < m - 1;
    edge += (so ? s[q - m] : 0.0) + (no ? s[q + m] : 0.0);
    corner = ((so && w) ? s[q - m - 1] : 0.0) + ((so && e) ? s[q - m + 1] : 0.0) +
             ((no && w) ? s[q + m - 1] : 0.0) + ((no && e) ? s[q + m + 1] : 0.0);
  }
}

// Q1 elements: (M + tau K) v^n - ps_scale M ps at one point (ps = the slice
// before, or the wrapped last slice of P_eps, or null).
__device__ __forceinline__ double apply_row_q1(const double* __restrict__ vs,
                                               const double* __restrict__ ps, double ps_scale,
                                               long long q, int ix, int iy, const StencilGeom& g,
                                               double center) {
  double e, k;
  neighbour_sums(vs, q, ix, iy, g, e, k);
  double y = fma(g.ac, center, fma(g.ae, e, g.ak * k));
  if (ps != nullptr) {
    double pe, pk;
    neighbour_sums(ps, q, ix, iy, g, pe, pk);
    y = fma(-ps_scale, fma(g.mc, ps[q], fma(g.me, pe, g.mk * pk)), y);
  }
  return y;
}

// Q1 elements, two-step scheme: (r0 M + tau K) v^n + s1 M ps + s2 M ps2 at one
// point (ps, ps2 = the slices one and two back, wrapped or null).
__device__ __forceinline__ double apply_row_q1_p2(const double* __restrict__ vs,
                                                  const double* __restrict__ ps, double s1,
                                                  const double* __restrict__ ps2, double s2,
                                                  long long q, int ix, int iy, const StencilGeom& g,
                                                  double center) {
  double e, k;
  neighbour_sums(vs, q, ix, iy, g, e, k);
  double y = fma(g.ac, center, fma(g.ae, e, g.ak * k));
  if (ps != nullptr) {
    double pe, pk;
    neighbour_sums(ps, q, ix, iy, g, pe, pk);
    y = fma(s1, fma(g.mc, ps[q], fma(g.me, pe, g.mk * pk)), y);
  }
  if (ps2 != nullptr) {
    double pe, pk;
    neighbour_sums(ps2, q, ix, iy, g, pe, pk);
    y = fma(s2, fma(g.mc, ps2[q], fma(g.me, pe, g.mk * pk)), y);
  }
  return y;
}

// M u at one point (Q1 elements)
__device__ __forceinline__ double mass_row_q1(const double* __restrict__ us, long long q, int ix,
                                              int iy, const StencilGeom& g) {
  double e, k;
  neighbour_sums(us, q, ix, iy, g, e, k);
  return fma(g.mc, us[q], fma(g.me, e, g.mk * k));
}

// The operator a kernel instantiation applies: finite differences in 1D or
// 2D (constant or variable a), Q1 elements (1D or 2D), finite differences in 3D.
enum { kFD = 0, kQ1 = 1, kFD3 = 2 };

// point q of a slice as (ix, iy, iz): x fastest, rows of m points
template <int KIND>
__device__ __forceinline__ void decompose(long long q, const StencilGeom& g, int& ix, int& iy,
                                          int& iz) {
  if constexpr (KIND == kFD3) {
    const long long r = q / g.m;
    ix = (int)(q - r * g.m);
    iz = (int)(r / g.m);
    iy = (int)(r - (long long)iz * g.m);
  } else {
    iy = g.dim == 2 ? (int)(q / g.m) : 0;
    ix = (int)(q - (long long)iy * g.m);
    iz = 0;
  }
}

// (L v)^n at one point: c (alpha v - sum of neighbours) - v^{n-1}, which is
// (1 + 2 dim c) v - c (sum) - v^{n-1} in 3 FP64 adds and 2 FMAs (2D).
__device__ __forceinline__ double apply_row(const double* __restrict__ vs, long long q, int ix,
                                            int iy, int iz, const StencilGeom& g, double center,
                                            double prev) {
  if (g.kc != nullptr) {   // variable coefficient: v + tau K v - v^{n-1}
    const long long J = g.J;
    double t = fma(g.kc[q], center, center - prev);
    if (ix > 0) t = fma(-g.kc[J + q], vs[q - 1], t);
    if (ix < g.m - 1) t = fma(-g.kc[2 * J + q], vs[q + 1], t);
    if (iy > 0) t = fma(-g.kc[3 * J + q], vs[q - g.m], t);
    if (iy < g.m - 1) t = fma(-g.kc[4 * J + q], vs[q + g.m], t);
    return t;
  }
  double nb = (ix > 0 ? vs[q - 1] : 0.0) + (ix < g.m - 1 ? vs[q + 1] : 0.0);
  if (g.dim == 2) nb += (iy > 0 ? vs[q - g.m] : 0.0) + (iy < g.m - 1 ? vs[q + g.m] : 0.0);
  return fma(g.c, fma(g.alpha, center, -nb), -prev);
}

// 3D finite differences (7-point): (1 + 6c) v - c (sum of the 6 neighbours) - v^{n-1}
__device__ __forceinline__ double apply_row3(const double* __restrict__ vs, long long q, int ix,
                                             int iy, int iz, const StencilGeom& g, double center,
                                             double prev) {
  const long long m2 = (long long)g.m * g.m;
  const double nb = (ix > 0 ? vs[q - 1] : 0.0) + (ix < g.m - 1 ? vs[q + 1] : 0.0) +
                    (iy > 0 ? vs[q - g.m] : 0.0) + (iy < g.m - 1 ? vs[q + g.m] : 0.0) +
                    (iz > 0 ? vs[q - m2] : 0.0) + (iz < g.m - 1 ? vs[q + m2] : 0.0);
  return fma(g.c, fma(g.alpha, center, -nb), -prev);
}

// the row of L (or P_eps without the wrap) of kernel kind KIND and P-step
// scheme at one point; ps, ps2 = the slices one and two back (Q1 only; null
// before the first slice); prev, prev2 = v^{n-1}, v^{n-2} at the point (FD)
template <int KIND, int P>
__device__ __forceinline__ double row_of(const double* __restrict__ vs,
                                         const double* __restrict__ ps,
                                         const double* __restrict__ ps2, long long q, int ix,
                                         int iy, int iz, const StencilGeom& g, double center,
                                         double prev, double prev2) {
  if constexpr (P == 2) {
    static_assert(KIND != kFD3, "the two-step scheme is 1D or 2D");
    if constexpr (KIND == kQ1) {
      return apply_row_q1_p2(vs, ps, g.r1, ps2, g.r2, q, ix, iy, g, center);
    } else {
      double nb = (ix > 0 ? vs[q - 1] : 0.0) + (ix < g.m - 1 ? vs[q + 1] : 0.0);
      if (g.dim == 2) nb += (iy > 0 ? vs[q - g.m] : 0.0) + (iy < g.m - 1 ? vs[q + g.m] : 0.0);
      return fma(g.c, fma(g.alpha, center, -nb), fma(g.r1, prev, g.r2 * prev2));
    }
  } else if constexpr (KIND == kQ1) {
    return apply_row_q1(vs, ps, 1.0, q, ix, iy, g, center);
  } else if constexpr (KIND == kFD3) {
    return apply_row3(vs, q, ix, iy, iz, g, center, prev);
  } else {
    return apply_row(vs, q, ix, iy, iz, g, center, prev);
  }
}

// slice n - j of v for row n, or the slice wrapped around by P_eps (corner
// != 0) with *scale multiplied by corner; null when there is none
__device__ __forceinline__ const double* back_slice(const double* __restrict__ v, int n, int j,
                                                    const StencilGeom& g, double corner,
                                                    double& scale) {
  if (n - j >= 0) return v + (long long)(n - j) * g.J;
  if (corner == 0.0) return nullptr;
  scale *= corner;
  return v + (long long)(n - j + g.N) * g.J;
}

// y = L v (corner = 0) or y = P_eps v (corner = eps), times *out_scale if given.
template <int KIND, int P>
__global__ void __launch_bounds__(kStencilThreads)
apply_L_kernel(const double* __restrict__ v, double* __restrict__ y, StencilGeom g,
               double corner, const double* __restrict__ out_scale) {
  const long long q = (long long)blockIdx.x * kStencilThreads + threadIdx.x;
  if (q >= g.J) return;
  const int n0 = blockIdx.y * kTimeChunk;
  const int n1 = min(g.N, n0 + kTimeChunk);
  int ix, iy, iz;
  decompose<KIND>(q, g, ix, iy, iz);
  // v^{n0-1} and v^{n0-2} at this point, wrapped around (times corner) by P_eps
  double prev = n0 > 0 ? v[(long long)(n0 - 1) * g.J + q]
                       : (corner != 0.0 ? corner * v[(long long)(g.N - 1) * g.J + q] : 0.0);
  double prev2 = 0.0;
  if constexpr (P == 2) {
    prev2 = n0 > 1 ? v[(long long)(n0 - 2) * g.J + q]
                   : (corner != 0.0 ? corner * v[(long long)(n0 - 2 + g.N) * g.J + q] : 0.0);
  }
  const double sc = out_scale ? out_scale[0] : 1.0;
  for (int n = n0; n < n1; ++n) {
    const double* vs = v + (long long)n * g.J;
    const double center = vs[q];
    double r;
    if constexpr (KIND == kQ1 && P == 2) {
      double s1 = g.r1, s2 = g.r2;
      const double* ps = back_slice(v, n, 1, g, corner, s1);
      const double* ps2 = back_slice(v, n, 2, g, corner, s2);
      r = apply_row_q1_p2(vs, ps, s1, ps2, s2, q, ix, iy, g, center);
    } else if constexpr (KIND == kQ1) {
      const double* ps = n > 0 ? vs - g.J : (corner != 0.0 ? v + (long long)(g.N - 1) * g.J : nullptr);
      r = apply_row_q1(vs, ps, n > 0 ? 1.0 : corner, q, ix, iy, g, center);
    } else {
      r = row_of<KIND, P>(vs, nullptr, nullptr, q, ix, iy, iz, g, center, prev, prev2);
    }
    y[(long long)n * g.J + q] = out_scale ? sc * r : r;
    prev2 = prev;
    prev = center;
  }
}

// w = L z and, for v < NV, the block sums of V_v . w: the first Gram-Schmidt
// pass fused with the operator.  A fixed grid walks the (256-point tile, time
// chunk) pairs in a fixed order, so the partial sums are reproducible.
template <int NV, int KIND, int P>
__global__ void __launch_bounds__(kStencilThreads)
stencil_dots_kernel(const double* __restrict__ z, double* __restrict__ w, StencilGeom g, VecList V,
                    const double* __restrict__ vshift, const double* __restrict__ sshift,
                    double* __restrict__ partials) {
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
  double accn = 0.0;
  const double ss = vshift ? sshift[0] : 0.0;
  const long long jt = (g.J + kStencilThreads - 1) / kStencilThreads;
  const long long tiles = jt * ((g.N + kTimeChunk - 1) / kTimeChunk);
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const long long q = (t % jt) * kStencilThreads + threadIdx.x;
    if (q >= g.J) continue;
    const int n0 = (int)(t / jt) * kTimeChunk;
    const int n1 = min(g.N, n0 + kTimeChunk);
    int ix, iy, iz;
    decompose<KIND>(q, g, ix, iy, iz);
    double prev = n0 > 0 ? z[(long long)(n0 - 1) * g.J + q] : 0.0;
    double prev2 = (P == 2 && n0 > 1) ? z[(long long)(n0 - 2) * g.J + q] : 0.0;
    for (int n = n0; n < n1; ++n) {
      const double* zs = z + (long long)n * g.J;
      const double center = zs[q];
      const long long o = (long long)n * g.J + q;
      double y = row_of<KIND, P>(zs, n > 0 ? zs - g.J : nullptr, n > 1 ? zs - 2 * g.J : nullptr, q,
                                 ix, iy, iz, g, center, prev, prev2);
      if (vshift) y = fma(-ss, vshift[o], y);
      w[o] = y;
      prev2 = prev;
      prev = center;
      accn = fma(y, y, accn);
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = fma(V.v[v][o], y, acc[v]);
    }
  }
  __shared__ double red[kStencilThreads / 32][NV + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    double s = acc[v];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) red[warp][v] = s;
  }
  for (int off = 16; off > 0; off >>= 1) accn += __shfl_down_sync(0xffffffffu, accn, off);
  if (lane == 0) red[warp][NV] = accn;
  __syncthreads();
  if ((int)threadIdx.x <= NV) {
    double s = 0.0;
#pragma unroll
    for (int wi = 0; wi < kStencilThreads / 32; ++wi) s += red[wi][threadIdx.x];
    partials[(long long)threadIdx.x * gridDim.x + blockIdx.x] = s;   // row NV: sum of w^2
  }
}

// r = f - L u (u == nullptr: r = f)
template <int KIND, int P>
__global__ void __launch_bounds__(kStencilThreads)
residual_kernel(const double* __restrict__ f, const double* __restrict__ u,
                double* __restrict__ r, StencilGeom g) {
  const long long q = (long long)blockIdx.x * kStencilThreads + threadIdx.x;
  if (q >= g.J) return;
  const int n0 = blockIdx.y * kTimeChunk;
  const int n1 = min(g.N, n0 + kTimeChunk);
  int ix, iy, iz;
  decompose<KIND>(q, g, ix, iy, iz);
  if (u == nullptr) {
    for (int n = n0; n < n1; ++n) r[(long long)n * g.J + q] = f[(long long)n * g.J + q];
    return;
  }
  double prev = n0 > 0 ? u[(long long)(n0 - 1) * g.J + q] : 0.0;
  double prev2 = (P == 2 && n0 > 1) ? u[(long long)(n0 - 2) * g.J + q] : 0.0;
  for (int n = n0; n < n1; ++n) {
    const double* us = u + (long long)n * g.J;
    const double center = us[q];
    const long long o = (long long)n * g.J + q;
    r[o] = f[o] - row_of<KIND, P>(us, n > 0 ? us - g.J : nullptr, n > 1 ? us - 2 * g.J : nullptr,
                                  q, ix, iy, iz, g, center, prev, prev2);
    prev2 = prev;
    prev = center;
  }
}

// Block sums of (f - L u)^2 and f^2 for RES (Sec. 5).  One partial pair per
// block, reduced in a fixed order by finish_norms_kernel: deterministic.
template <int KIND, int P>
__global__ void __launch_bounds__(kStencilThreads)
residual_norms_kernel(const double* __restrict__ f, const double* __restrict__ u,
                      double* __restrict__ partials, StencilGeom g) {
  const long long q = (long long)blockIdx.x * kStencilThreads + threadIdx.x;
  double rr = 0.0, ff = 0.0;
  if (q < g.J) {
    const int n0 = blockIdx.y * kTimeChunk;
    const int n1 = min(g.N, n0 + kTimeChunk);
    int ix, iy, iz;
    decompose<KIND>(q, g, ix, iy, iz);
    double prev = n0 > 0 ? u[(long long)(n0 - 1) * g.J + q] : 0.0;
    double prev2 = (P == 2 && n0 > 1) ? u[(long long)(n0 - 2) * g.J + q] : 0.0;
    for (int n = n0; n < n1; ++n) {
      const double* us = u + (long long)n * g.J;
      const double center = us[q];
      const long long o = (long long)n * g.J + q;
      const double fo = f[o];
      const double r = fo - row_of<KIND, P>(us, n > 0 ? us - g.J : nullptr,
                                            n > 1 ? us - 2 * g.J : nullptr, q, ix, iy, iz, g,
                                            center, prev, prev2);
      rr += r * r;
      ff += fo * fo;
      prev2 = prev;
      prev = center;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    rr += __shfl_down_sync(0xffffffffu, rr, off);
    ff += __shfl_down_sync(0xffffffffu, ff, off);
  }
  __shared__ double s_rr[kStencilThreads / 32], s_ff[kStencilThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    s_rr[warp] = rr;
    s_ff[warp] = ff;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < kStencilThreads / 32; ++w) {
      a += s_rr[w];
      b += s_ff[w];
    }
    const long long blk = (long long)blockIdx.y * gridDim.x + blockIdx.x;
    partials[2 * blk] = a;
    partials[2 * blk + 1] = b;
  }
}

// fslot >= 0: ||f|| is scal[fslot] already; host != null: the scalars to the host's copy
__global__ void finish_norms_kernel(const double* __restrict__ partials, long long nblk,
                                    double* scal, int slot, int fslot, double* host) {
  __shared__ double s_a[256], s_b[256];
  double a = 0.0, b = 0.0;
  for (long long i = threadIdx.x; i < nblk; i += blockDim.x) {
    a += partials[2 * i];
    b += partials[2 * i + 1];
  }
  s_a[threadIdx.x] = a;
  s_b[threadIdx.x] = b;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      s_a[threadIdx.x] += s_a[threadIdx.x + s];
      s_b[threadIdx.x] += s_b[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    scal[slot] = sqrt(s_a[0]);
    scal[slot + 1] = fslot >= 0 ? scal[fslot] : sqrt(s_b[0]);
  }
  if (host != nullptr) {
    __syncthreads();
    if ((int)threadIdx.x < kScalSlots) host[threadIdx.x] = scal[threadIdx.x];
  }
}

// f = tau fsrc, plus M u0 in slice 1 (Sec. 2; M = I for finite differences);
// two-step scheme: plus rhs1 M u0 in slice 1 and rhs2 M u0 in slice 2.
__global__ void build_rhs_kernel(const double* __restrict__ u0, const double* __restrict__ fsrc,
                                 double* __restrict__ f, StencilGeom g, double tau) {
  const long long U = g.J * g.N;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < U;
       i += (long long)gridDim.x * blockDim.x) {
    double v = tau * fsrc[i];
    const double coef = i < g.J ? g.rhs1 : (i < 2 * g.J ? g.rhs2 : 0.0);
    if (coef != 0.0) {
      const long long q = i < g.J ? i : i - g.J;
      double mu;
      if (g.q1) {
        int ix, iy, iz;
        decompose<kQ1>(q, g, ix, iy, iz);
        mu = mass_row_q1(u0, q, ix, iy, g);
      } else {
        mu = u0[q];
      }
      v = coef == 1.0 ? v + mu : fma(coef, mu, v);
    }
    f[i] = v;
  }
}

// ---------------------------------------------------------------- fixed point
// The rows of L in 64-bit fixed point (bec_fx.cuh) with a constant coefficient:
// finite differences in 2D and 3D, Q1 elements in 2D.
//
// GB300 issues 2 FP64 operations a clock and SM: the 5 (2D) or 7 (3D) of a row
// bound the kernels above, whose vectors' traffic takes a quarter of that time.
// Here a row is integer work: L v = c (2 dim v - sum of neighbours) + v - v^{n-1}
// with the differences exact, one product by c and one conversion to FP64; the
// FP64 pipe keeps only what follows (the shift, the dots, the norms).
//
// A warp owns 32 columns and kFxRows rows of one slice (3D: of one plane) and
// walks a chunk of time steps.  A lane converts its rows and the two beside
// them once and gets its x neighbours by shuffle; only the edge lanes load one
// more value a row.  The unit is a power of two from the largest value of the
// tile in the steps that the row takes (v^n, v^{n-1}; two-step scheme: v^{n-2}),
// so that |v| < 2^59: the error is below 2^-55 c times that value.  The steps
// before v^n are carried as bit patterns and converted in each row's own unit: an
// integer in the unit of the row before would have lost bits to v^{n-2}.  Values
// that are not finite, leave the range or are below 2^-951 go through the FP64 row.
// Measured at 255^2 x 256: w = L z - s v with 1 and 2 dots 158 us on average
// (FP64 rows: 287), ||f - L u|| 127 us (300); what bounds them now is the FP64
// pipe again (2 operations and one a dot), 70 to 80 % busy.  Converting v^{n-1}
// again only where the unit changes costs more branches than it saves (183 us).
//
// Q1 rows take six products, three of them by M, which the next step's row
// subtracts: a lane keeps M v^{n-1} instead of the values.  At 127^2 x 64 (1M
// unknowns) L v takes 20 us (FP64 rows: 56), ||f - L u|| 24 us (61).
//
// Variable coefficients keep the FP64 rows: five products on the tile's own
// scale took w and its dots from 390 to 340 us at 255^2 x 256 (3 % of a
// multigrid solve), and the other rounding of L moved solutions of the FP32
// multigrid solves by up to 2e-10.
constexpr int kFxRows = 4;
constexpr int kFxTiny = fx::kFxMin + 1081;   // smallest exponent field that fills the least unit
constexpr int kFxDotVecs = 8;        // vectors a fused launch takes; more go to dots_kernel

struct FxStencil {
  fx::W64 cm;      // c = cm 2^-63 2^ce
  fx::W64 wa[3], wm[3];   // Q1: centre, edge, corner of M + tau K and of M, times 2^(63 - ce)
  int ce;
  int kc, ke;             // Q1: exponents of 1.5 2^ce over the centre and the edge of M + tau K
  int chunk;       // time steps of a tile
  int xt, yg, planes;   // tiles in x, row groups, planes (3D: m)
  int tiles;
};

enum { kModeDots = 0, kModeNorms = 1, kModeApply = 2, kModeResidual = 3 };

// the FP64 row at point q of the slice vs = v^n
template <int KIND, int P>
__device__ __noinline__ double fx_slow_row(const double* __restrict__ vs, long long q, int ix, int iy, int iz,
                                           int n, const StencilGeom& g) {
  return row_of<KIND, P>(vs, KIND == kQ1 && n > 0 ? vs - g.J : nullptr, nullptr, q, ix, iy, iz, g, vs[q],
                         n > 0 ? vs[q - g.J] : 0.0,
                         P == 2 && n > 1 ? vs[q - 2 * g.J] : 0.0);
}

// Finite differences: which of the lane's rows (mask) are below T (high words of the
// bit patterns) in all their own values and not zero in all, from memory; `time`:
// v^n and the steps before it count, not the neighbours.  These rows in FP64.
template <int KIND, int P>
__device__ __noinline__ void fx_small_rows(double* y, unsigned mask, int T, bool time, const double* __restrict__ vs,
                                           long long q, int ix, int iy, int iz, int n, const StencilGeom& g) {
  auto key = [](double v) { return fx::d_habs(fx::d_bits(v)) | ((unsigned)fx::d_bits(v) != 0); };
  for (int r = 0; r < kFxRows; ++r) {
    if (!(mask >> r & 1)) continue;
    const double* p = vs + q + (long long)r * g.m;
    const int c = key(p[0]), m1 = g.m - 1;
    int near = max(c, max(ix > 0 ? key(p[-1]) : 0, ix < m1 ? key(p[1]) : 0));
    near = max(near, max(iy + r > 0 ? key(p[-g.m]) : 0, iy + r < m1 ? key(p[g.m]) : 0));
    if constexpr (KIND == kFD3) {
      const long long m2 = (long long)g.m * g.m;
      near = max(near, max(iz > 0 ? key(p[-m2]) : 0, iz < m1 ? key(p[m2]) : 0));
    }
    const int back = max(n > 0 ? key(p[-g.J]) : 0, P == 2 && n > 1 ? key(p[-2 * g.J]) : 0);
    if (max(near, back) != 0 && (time ? max(c, back) : near) < T)
      y[r] = fx_slow_row<KIND, P>(vs, q + (long long)r * g.m, ix, iy + r, iz, n, g);
  }
}

// OWN: every row is as accurate as in FP64 for its own values.  Without it a row
// can hold fewer bits than that where its values are more than 6 bits below the
// tile's largest: what the solver takes from the rows are norms, dots and Krylov
// vectors, and in norm the error is below that of FP64 rows.  With OWN, 6 % of the
// tile's steps of a smooth solution have such rows; all of a solve's passes so cost
// 5 to 25 % more each (dots at 255^2 x 256 173 us instead of 158, Q1 rows at 127^2 x
// 64 31 instead of 20), so only bec_apply_A, whose rows a program sees, has it.
template <int KIND, int P, bool OWN>
struct FxRow {
  static constexpr int R = kFxRows;
  static constexpr bool D3 = KIND == kFD3, Q1 = KIND == kQ1;
  static constexpr int ER = Q1 ? R + 2 : R;   // rows whose left and right ends are wanted
  // one slice's values of the tile, as bit patterns (zeros outside the domain)
  struct Raw {
    fx::u64 b[R + 2];        // the lane's column: the row below, the rows, the row above
    fx::u64 edge;            // lane r < ER: left of row r (Q1: r - 1); lane ER + r: right of it
    fx::u64 d[D3 ? R : 1], u[D3 ? R : 1];   // 3D: the planes below and above
  };
  int m, lane, x, y0, z0, rows;
  unsigned in;               // which of b[] lie inside the domain; bit 31: the edge value
  long long q0, eo;          // the lane's first row; its edge value's point
  // v^{n-1} (and v^{n-2}) of the rows as bit patterns: every row takes them in its
  // own unit.  Q1: M v^{n-1} in the unit 2^Fp of v^{n-1} alone.
  fx::i64 prev[R], prev2[P == 2 ? R : 1];
  int Fp, ep, ep2;           // Q1: unit of prev; largest exponent fields of v^{n-1}, v^{n-2}

  __device__ __forceinline__ void start(const StencilGeom& g, const FxStencil& f, int t, int ln) {
    lane = ln;
    m = g.m;
    const int a = t / f.xt, x0 = (t - a * f.xt) * 32;
    z0 = D3 ? a / f.yg : 0;
    y0 = (a - z0 * f.yg) * R;
    x = x0 + lane;
    rows = min(R, m - y0);
    q0 = ((long long)z0 * m + y0) * m + x;
    in = 0;
    if (x < m) {
      in = ((1u << rows) - 1u) << 1;
      if (y0 > 0) in |= 1u;
      if (y0 + rows < m) in |= 1u << (rows + 1);
    }
    const int er = lane % ER - (Q1 ? 1 : 0), ex = lane < ER ? x0 - 1 : x0 + 32;
    if (lane < 2 * ER && er < rows + (Q1 ? 1 : 0) && y0 + er >= 0 && y0 + er < m && ex >= 0 && ex < m)
      in |= 1u << 31;
    eo = ((long long)z0 * m + y0 + er) * m + ex;
  }
  __device__ __forceinline__ bool row_in(int r) const { return in >> (r + 1) & 1; }
  __device__ __forceinline__ void load(const double* __restrict__ vs, Raw& w) const {
    const double* p = vs + q0;
#pragma unroll
    for (int r = 0; r < R + 2; ++r) w.b[r] = in >> r & 1 ? fx::d_bits(p[(r - 1) * m]) : 0;
    w.edge = in >> 31 ? fx::d_bits(vs[eo]) : 0;
    if constexpr (D3) {
      const long long m2 = (long long)m * m;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        w.d[r] = row_in(r) && z0 > 0 ? fx::d_bits(p[r * m - m2]) : 0;
        w.u[r] = row_in(r) && z0 + 1 < m ? fx::d_bits(p[r * m + m2]) : 0;
      }
    }
  }
  // the centre values of a slice (zeros where there is none)
  __device__ __forceinline__ void load_prev(const double* __restrict__ vs, fx::i64 (&pv)[R], int& e) {
    int h = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const fx::u64 b = vs != nullptr && row_in(r) ? fx::d_bits(vs[q0 + r * m]) : 0;
      pv[r] = (fx::i64)b;
      h = max(h, fx::d_habs(b));
    }
    e = (int)__reduce_max_sync(0xffffffffu, (unsigned)h) >> 20;
  }
  // Q1: visit(r, centre, sum of the 4 edge neighbours, of the 4 corners) for the
  // rows of a slice, in the unit 2^F
  template <typename Visit>
  __device__ __forceinline__ void q1_rows(const Raw& w, int F, Visit visit) const {
    using fx::i64;
    const i64 edge = fx::d_to_fx(w.edge, F);
    auto ends = [&](i64 c, int r) {                       // left plus right of row r - 1
      i64 le = __shfl_up_sync(0xffffffffu, c, 1), ri = __shfl_down_sync(0xffffffffu, c, 1);
      const i64 ed = __shfl_sync(0xffffffffu, edge, lane < 16 ? r : ER + r);
      if (lane == 0) le = ed;
      if (lane == 31) ri = ed;
      return le + ri;
    };
    i64 below = fx::d_to_fx(w.b[0], F), c = fx::d_to_fx(w.b[1], F);
    i64 hb = ends(below, 0), h = ends(c, 1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const i64 above = fx::d_to_fx(w.b[r + 2], F), ha = ends(above, r + 2);
      visit(r, c, h + (below + above), hb + ha);
      below = c;
      c = above;
      hb = h;
      h = ha;
    }
  }
  __device__ __forceinline__ int q1_max(const Raw& w) const {
    int h = fx::d_habs(w.edge);
#pragma unroll
    for (int r = 0; r < R + 2; ++r) h = max(h, fx::d_habs(w.b[r]));
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)h) >> 20;
  }
  static __device__ __forceinline__ fx::i64 q1_form(const fx::W64 (&k)[3], fx::i64 c, fx::i64 e, fx::i64 d) {
    return (fx::mul64(c, k[0]) + fx::mul64(e, k[1])) + fx::mul64(d, k[2]);
  }
  // prev = M times the slice vs
  __device__ __forceinline__ void load_prev_q1(const double* __restrict__ vs, const FxStencil& f) {
    Raw w;
    if (vs != nullptr) load(vs, w);
    else w = Raw{};
    ep = q1_max(w);
    Fp = max(ep - 1081, fx::kFxMin);
    q1_rows(w, Fp, [&](int r, fx::i64 c, fx::i64 e, fx::i64 d) { prev[r] = q1_form(f.wm, c, e, d); });
  }
  // y = rows of (M + tau K) v^n - M v^{n-1}.  Each part is formed in the unit of
  // its own slice (|v| < 2^59 and |coefficient| < 2^63: below 2^61.2); the finer
  // one is rounded to the other's unit, so that a row sees its own operands only.
  __device__ __forceinline__ void step_q1(const Raw& w, const double* __restrict__ vs, const StencilGeom& g,
                                          const FxStencil& f, int n, double (&y)[R]) {
    const int e = q1_max(w), em = max(e, ep);
    const int F = max(e - 1081, fx::kFxMin), G = max(F, Fp) + f.ce + 1;
    const int da = min(max(Fp - F, 0), 63), dp = min(max(F - Fp, 0), 63);
    const fx::i64 ra = da > 0 ? 1LL << (da - 1) : 0, rp = dp > 0 ? 1LL << (dp - 1) : 0;
    // else all rows in FP64: not finite, out of range, or too small to fill the unit
    const bool plain = em != 0x7FF && fx::fx_normal(G) && em >= kFxTiny;
    int low = 0x7FFFFFFF;                                 // smallest of the rows' larger parts
    q1_rows(w, F, [&](int r, fx::i64 c, fx::i64 eg, fx::i64 d) {
      const fx::i64 A = fx::shr(q1_form(f.wa, c, eg, d) + ra, da), M = fx::shr(prev[r] + rp, dp);
      prev[r] = q1_form(f.wm, c, eg, d);
      if constexpr (OWN) {
        const int q = max(high(A), high(M));
        low = min(low, row_in(r) ? q : 0x7FFFFFFF);
      }
      if (plain) y[r] = fx::fx_to_d(A - M, G);
    });
    if (!plain) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        y[r] = row_in(r) ? fx_slow_row<KIND, P>(vs, q0 + r * m, x, y0 + r, z0, n, g) : 0.0;
    } else if (OWN && low < 1 << 21) {
      // An FP64 row's error is about 2^-53 of each of its parts and products, a row's
      // here about a unit: where none of those looked at reaches 2^53 units, the row
      // is taken in FP64.
      const int T = max(F, Fp) + 1076, Tc = min(T + f.kc, 2047) << 20, Te = min(T + f.ke, 2047) << 20;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (row_in(r) && fx::d_habs(w.b[r + 1]) < Tc && max(fx::d_habs(w.b[r]), fx::d_habs(w.b[r + 2])) < Te)
          y[r] = fx_slow_row<KIND, P>(vs, q0 + r * m, x, y0 + r, z0, n, g);
    }
    ep = e;
    Fp = F;
  }
  // high word of |v|, less one below zero
  static __device__ __forceinline__ int high(fx::i64 v) { return (int)(v >> 32) ^ (int)(v >> 63); }
  // y = row values of the slice vs = v^n, whose values are in w
  __device__ __forceinline__ void step(const Raw& w, const double* __restrict__ vs, const StencilGeom& g,
                                       const FxStencil& f, int n, double (&y)[R]) {
    using fx::i64;
    int h = fx::d_habs(w.edge);
#pragma unroll
    for (int r = 0; r < R + 2; ++r) h = max(h, fx::d_habs(w.b[r]));
    if constexpr (D3) {
#pragma unroll
      for (int r = 0; r < R; ++r) h = max(h, max(fx::d_habs(w.d[r]), fx::d_habs(w.u[r])));
    }
    const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)h) >> 20;
    const int em = max(max(e, ep), P == 2 ? ep2 : 0);
    const int F = max(em - 1081, fx::kFxMin);            // |v| < 2^(em - 1022) = 2^(F + 59)
    const int s = f.ce + 1;                               // c lap = mul64(lap, cm) 2^s
    const int G = F + max(s, 0);
    if constexpr (P == 2) ep2 = ep;
    ep = e;
    // not finite, out of range, or too small to fill the unit
    if (em == 0x7FF || !fx::fx_normal(G) || em < kFxTiny) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        y[r] = row_in(r) ? fx_slow_row<KIND, P>(vs, q0 + r * m, x, y0 + r, z0, n, g) : 0.0;
        if constexpr (P == 2) prev2[r] = prev[r];
        prev[r] = (i64)w.b[r + 1];
      }
      return;
    }
    // OWN: a row whose own values are all more than 6 bits below the largest holds fewer
    // than FP64's 53: it is taken in FP64.  The values that count are v^n and its
    // neighbours, or with c < 1/4, where the error is that of v^n - v^{n-1}, those
    // two.  Looked at first are a part of them, mostly enough: a lane's own, then the
    // centres beside it.
    const int T = (F + 1076) << 20;                       // 2^(F + 53)
    bool small = false;
    if constexpr (OWN) {
      int low = 0x7FFFFFFF;
      if (s >= 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int q = max(max(fx::d_habs(w.b[r]), fx::d_habs(w.b[r + 1])), fx::d_habs(w.b[r + 2]));
          low = min(low, row_in(r) ? q : 0x7FFFFFFF);
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
          low = min(low, row_in(r) ? max(fx::d_habs(w.b[r + 1]), fx::d_habs((fx::u64)prev[r])) : 0x7FFFFFFF);
      }
      small = low < T;
      if (__any_sync(0xffffffffu, small) && s >= 0) {     // the centres beside the lane's
        int c = 0x7FFFFFFF;
#pragma unroll
        for (int r = 0; r < R; ++r) c = min(c, row_in(r) ? fx::d_habs(w.b[r + 1]) : 0x7FFFFFFF);
        if (x >= m) c = 0;
        const int side = max(__shfl_up_sync(0xffffffffu, c, 1), __shfl_down_sync(0xffffffffu, c, 1));
        small = small && side < T;                        // every lane takes part in the shuffles
      }
    }
    // shifts round to nearest: a bias of even a small part of a unit, the same at
    // every point, would come back from L^{-1} many times larger
    const i64 rnd = s == 0 ? 0 : 1LL << (min(abs(s), 60) - 1);
    const i64 edge = fx::d_to_fx(w.edge, F);
    i64 below = fx::d_to_fx(w.b[0], F), c = fx::d_to_fx(w.b[1], F);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const i64 above = fx::d_to_fx(w.b[r + 2], F);
      i64 le = __shfl_up_sync(0xffffffffu, c, 1), ri = __shfl_down_sync(0xffffffffu, c, 1);
      const i64 ed = __shfl_sync(0xffffffffu, edge, lane < 16 ? r : R + r);
      if (lane == 0) le = ed;
      if (lane == 31) ri = ed;
      i64 lap = (c << 2) - ((le + ri) + (below + above));
      if constexpr (D3) lap += (c << 1) - (fx::d_to_fx(w.d[r], F) + fx::d_to_fx(w.u[r], F));
      const i64 t = fx::mul64(lap, f.cm);
      i64 Y;
      if constexpr (P == 2) {                             // (3 v - 4 v' + v'') / 2
        const i64 d = 3 * c - 4 * fx::d_to_fx((fx::u64)prev[r], F) + fx::d_to_fx((fx::u64)prev2[r], F);
        Y = s >= 0 ? t + fx::shr(d + (1LL << s), s + 1) : fx::shr(t + rnd, -s) + ((d + 1) >> 1);
        prev2[r] = prev[r];
      } else {
        const i64 d = c - fx::d_to_fx((fx::u64)prev[r], F);
        Y = s >= 0 ? t + fx::shr(d + rnd, s) : fx::shr(t + rnd, -s) + d;
      }
      prev[r] = (i64)w.b[r + 1];
      y[r] = fx::fx_to_d(Y, G);
      below = c;
      c = above;
    }
    if (small) {
      double t[R];                                        // in memory, y stays in registers
#pragma unroll
      for (int r = 0; r < R; ++r) t[r] = y[r];
      fx_small_rows<KIND, P>(t, in >> 1 & ((1u << R) - 1u), T, s < 0, vs, q0, x, y0, z0, n, g);
#pragma unroll
      for (int r = 0; r < R; ++r) y[r] = t[r];
    }
  }
};

// z: the vector the rows apply to.  kModeDots: w = L z - s vshift, partials as
// stencil_dots_kernel (LAST: vshift is V_{NV-1}); kModeNorms: partials as
// residual_norms_kernel (aux = f; LAST: without f^2); kModeApply: w = L z (times *sshift if
// given); kModeResidual: w = aux - L z.
template <int MODE, int NV, bool LAST, int KIND, int P, bool OWN>
__global__ void __launch_bounds__(kStencilThreads, NV <= 2 && KIND == kFD ? 3 : 2)
stencil_fx_kernel(const double* __restrict__ z, const double* __restrict__ aux, double* __restrict__ w,
                  StencilGeom g, FxStencil f, VecList V, const double* __restrict__ vshift,
                  const double* __restrict__ sshift, double* __restrict__ partials) {
  using Row = FxRow<KIND, P, OWN>;
  constexpr int R = kFxRows, NA = MODE == kModeDots ? NV + 1 : 2;
  double acc[NA];
#pragma unroll
  for (int v = 0; v < NA; ++v) acc[v] = 0.0;
  const int lane = threadIdx.x & 31;
  const double ss = sshift ? sshift[0] : (MODE == kModeApply ? 1.0 : 0.0);
  const int wstep = gridDim.x * (kStencilThreads / 32), per = f.xt * f.yg * f.planes;
  Row row;
  for (int t = blockIdx.x * (kStencilThreads / 32) + (threadIdx.x >> 5); t < f.tiles; t += wstep) {
    const int tc = t / per;
    row.start(g, f, t - tc * per, lane);
    const int n0 = tc * f.chunk, n1 = min(g.N, n0 + f.chunk);
    const double* zs = z + (long long)n0 * g.J;
    typename Row::Raw cur, nxt;
    row.load(zs, cur);
    if constexpr (Row::Q1) row.load_prev_q1(n0 > 0 ? zs - g.J : nullptr, f);
    else row.load_prev(n0 > 0 ? zs - g.J : nullptr, row.prev, row.ep);
    if constexpr (P == 2)
      row.load_prev(n0 > 1 ? zs - 2 * g.J : nullptr, row.prev2, row.ep2);
    long long o0 = (long long)n0 * g.J + row.q0;
    for (int n = n0; n < n1; ++n) {
      // the next slice's values and this one's other operands are on their way
      // while this slice is worked on
      if (n + 1 < n1) row.load(zs + g.J, nxt);
      double a1[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a1[r] = 0.0;
        if (!row.row_in(r)) continue;
        if constexpr (MODE == kModeDots) a1[r] = LAST ? V.v[NV - 1][o0 + r * g.m] : vshift ? vshift[o0 + r * g.m] : 0.0;
        else if constexpr (MODE != kModeApply) a1[r] = aux[o0 + r * g.m];
      }
      double y[R];
      if constexpr (Row::Q1) row.step_q1(cur, zs, g, f, n, y);
      else row.step(cur, zs, g, f, n, y);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!row.row_in(r)) continue;
        const long long o = o0 + r * g.m;
        if constexpr (MODE == kModeDots) {
          const double a = fma(-ss, a1[r], y[r]);
          w[o] = a;
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = fma(LAST && v == NV - 1 ? a1[r] : V.v[v][o], a, acc[v]);
          acc[NV] = fma(a, a, acc[NV]);
        } else if constexpr (MODE == kModeNorms) {
          const double a = a1[r] - y[r];
          acc[0] = fma(a, a, acc[0]);
          if (!LAST) acc[1] = fma(a1[r], a1[r], acc[1]);
        } else if constexpr (MODE == kModeApply) {
          w[o] = sshift ? ss * y[r] : y[r];
        } else {
          w[o] = a1[r] - y[r];
        }
      }
      zs += g.J;
      o0 += g.J;
      cur = nxt;
    }
  }
  if constexpr (MODE == kModeDots || MODE == kModeNorms) {
    __shared__ double red[kStencilThreads / 32][NA];
    const int warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < NA; ++v) {
      double s = acc[v];
      for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
      if (lane == 0) red[warp][v] = s;
    }
    __syncthreads();
    if ((int)threadIdx.x < NA) {
      double s = 0.0;
#pragma unroll
      for (int wi = 0; wi < kStencilThreads / 32; ++wi) s += red[wi][threadIdx.x];
      // dots: row v of the partials; norms: pairs
      partials[MODE == kModeDots ? (long long)threadIdx.x * gridDim.x + blockIdx.x
                                 : 2LL * blockIdx.x + threadIdx.x] = s;
    }
  }
}

StencilGeom geom(const bec_problem* p) {
  StencilGeom g;
  g.J = p->J;
  g.m = p->m;
  g.N = p->N;
  g.dim = p->dim;
  // r0, r1, r2 of the time scheme (BDF1: 1, -1, 0; BDF2: 3/2, -2, 1/2)
  const bool bdf2 = p->desc.time_scheme == BEC_TIME_BDF2;
  const double r0 = bdf2 ? 1.5 : 1.0;
  g.r1 = bdf2 ? -2.0 : -1.0;
  g.r2 = bdf2 ? 0.5 : 0.0;
  // pre-start values taken equal to u^0: slice n gains -(r_n + ... + r_p) M u^0
  g.rhs1 = -(g.r1 + g.r2);
  g.rhs2 = -g.r2;
  g.c = p->tau * p->a / (p->h * p->h);
  g.alpha = (r0 + 2.0 * p->dim * g.c) / g.c;
  g.kc = p->kcoef;
  g.q1 = p->desc.space == BEC_SPACE_Q1;
  g.ac = g.ae = g.ak = g.mc = g.me = g.mk = 0.0;
  if (g.q1) {
    const double h = p->h, a = p->a, tau = p->tau;
    double kc, ke, kk;
    if (p->dim == 2) {   // M = h^2/36 [1 4 1; 4 16 4; 1 4 1], K = a/3 [-1 -1 -1; -1 8 -1; -1 -1 -1]
      g.mc = 16.0 * h * h / 36.0;
      g.me = 4.0 * h * h / 36.0;
      g.mk = h * h / 36.0;
      kc = 8.0 * a / 3.0;
      ke = -a / 3.0;
      kk = -a / 3.0;
    } else {             // M = h/6 [1 4 1], K = a/h [-1 2 -1]
      g.mc = 4.0 * h / 6.0;
      g.me = h / 6.0;
      g.mk = 0.0;
      kc = 2.0 * a / h;
      ke = -a / h;
      kk = 0.0;
    }
    g.ac = r0 * g.mc + tau * kc;
    g.ae = r0 * g.me + tau * ke;
    g.ak = r0 * g.mk + tau * kk;
  }
  return g;
}

int kind_of(const bec_problem* p) {
  if (p->desc.space == BEC_SPACE_Q1) return kQ1;
  return p->dim == 3 ? kFD3 : kFD;
}

// the kernel instantiation a problem uses: operator kind and time-scheme steps
enum { kVarFD = 0, kVarQ1, kVarFD3, kVarFD2, kVarQ12 };
int variant_of(const bec_problem* p) {
  const int k = kind_of(p);
  if (p->desc.time_scheme == BEC_TIME_BDF2) return k == kQ1 ? kVarQ12 : kVarFD2;
  return k == kQ1 ? kVarQ1 : (k == kFD3 ? kVarFD3 : kVarFD);
}

// LAUNCH(KIND, P) for the problem's variant
#define BEC_STENCIL_SWITCH(var, LAUNCH) \
  switch (var) {                         \
    case kVarQ1: LAUNCH(kQ1, 1); break;  \
    case kVarFD3: LAUNCH(kFD3, 1); break; \
    case kVarFD2: LAUNCH(kFD, 2); break; \
    case kVarQ12: LAUNCH(kQ1, 2); break; \
    default: LAUNCH(kFD, 1);             \
  }

template <int NV>
void stencil_dots_launch(int var, cudaStream_t st, const double* z, double* w,
                         const StencilGeom& g, const VecList& L, const double* vshift,
                         const double* sshift, double* partials) {
#define BEC_SD_LAUNCH(K, P)                                                      \
  stencil_dots_kernel<NV, K, P><<<kStencilDotBlocks, kStencilThreads, 0, st>>>( \
      z, w, g, L, vshift, sshift, partials)
  BEC_STENCIL_SWITCH(var, BEC_SD_LAUNCH)
#undef BEC_SD_LAUNCH
}

// The fixed-point rows take constant coefficients in 2D and 3D from 31 points a
// side (a warp's 32 columns are then nearly full): finite differences, and Q1
// elements (2D) with the one-step scheme.
bool fx_rows(const bec_problem* p) {
  return p->kcoef == nullptr && p->dim >= 2 && p->m >= 31 &&
         (p->desc.space == BEC_SPACE_FD || p->desc.time_scheme != BEC_TIME_BDF2);
}

// w = v 2^(63 - ce), |v| < 2^ce, as two words
fx::W64 fx_coef(double v, int ce) {
  long long w = (long long)std::ldexp(v, 63 - ce);
  if ((int)w == (int)0x80000000) ++w;             // the low word can be negated
  return fx::split64(w);
}

// Blocks of a launch, or fewer: 3 an SM.  The finite-difference kernels with up to
// 2 vectors are held to the registers for that (80 a thread, up to 120 bytes of
// them in local memory); the others take 118 to 128 and run 2 at a time, so that the
// last third of their blocks follows the first two.
constexpr int kFxBlocks = 3 * 152;
unsigned fx_stencil(const bec_problem* p, const StencilGeom& g, FxStencil& f) {
  int ce;
  const bool q1 = p->desc.space == BEC_SPACE_Q1;
  double top = g.c;
  if (q1) top = std::max(std::max(std::max(std::fabs(g.ac), std::fabs(g.ae)), std::fabs(g.ak)), g.mc);
  const double cm = std::frexp(top, &ce);
  if (cm > 0.9999999) ++ce;                       // next to 1: half of it
  const double wa[3] = {g.ac, g.ae, g.ak}, wm[3] = {g.mc, g.me, g.mk};
  for (int i = 0; i < 3; ++i) {
    f.wa[i] = fx_coef(wa[i], ce);
    f.wm[i] = fx_coef(wm[i], ce);
  }
  f.cm = fx_coef(q1 ? 0.0 : g.c, ce);
  f.kc = f.ke = 0;
  if (q1) {
    std::frexp(1.5 * std::ldexp(1.0, ce) / std::fabs(g.ac), &f.kc);
    const double ae = std::fabs(g.ae);
    if (ae > 1e-9 * top) std::frexp(1.5 * std::ldexp(1.0, ce) / ae, &f.ke);
    else f.ke = 1000;                             // edges never count
  }
  f.ce = ce;
  f.xt = (p->m + 31) / 32;
  f.yg = (p->m + kFxRows - 1) / kFxRows;
  f.planes = p->dim == 3 ? p->m : 1;
  const int per = f.xt * f.yg * f.planes;          // at most 2^23
  const long long warps = (long long)kFxBlocks * (kStencilThreads / 32);
  // the longest chunk that still gives every warp of the launch a tile
  f.chunk = 16;
  while (f.chunk > 1 && (long long)per * ((p->N + f.chunk - 1) / f.chunk) < warps) f.chunk /= 2;
  f.tiles = per * ((p->N + f.chunk - 1) / f.chunk);
  const int blocks = (f.tiles + kStencilThreads / 32 - 1) / (kStencilThreads / 32);
  return (unsigned)std::min(blocks, kFxBlocks);
}

template <int MODE, int NV, bool LAST = false, bool OWN = false>
void stencil_fx_launch(const bec_problem* p, unsigned grid, const double* z, const double* aux, double* w,
                       const StencilGeom& g, const FxStencil& f, const VecList& L, const double* vshift,
                       const double* sshift) {
#define BEC_SFX(K, P)                                                                       \
  stencil_fx_kernel<MODE, NV, LAST, K, P, OWN><<<grid, kStencilThreads, 0, p->stream>>>(               \
      z, aux, w, g, f, L, vshift, sshift, p->partials)
  if (p->dim == 3) BEC_SFX(kFD3, 1);
  else if (p->desc.space == BEC_SPACE_Q1) BEC_SFX(kQ1, 1);
  else if (p->desc.time_scheme == BEC_TIME_BDF2) BEC_SFX(kFD, 2);
  else BEC_SFX(kFD, 1);
#undef BEC_SFX
}

dim3 stencil_grid(const bec_problem* p) {
  return dim3((unsigned)((p->J + kStencilThreads - 1) / kStencilThreads),
              (unsigned)((p->N + kTimeChunk - 1) / kTimeChunk));
}

}  // namespace

long long stencil_blocks(const bec_problem* p) {
  const dim3 g = stencil_grid(p);
  return (long long)g.x * g.y;
}

bec_status launch_apply_L(bec_problem* p, const double* v, double* y, double corner,
                          const double* out_scale, bool own) {
  const StencilGeom g = geom(p);
  if (corner == 0.0 && fx_rows(p)) {
    FxStencil f;
    const unsigned grid = fx_stencil(p, g, f);
    BEC_LAUNCH_BEGIN(p);
    if (own)
      stencil_fx_launch<kModeApply, 1, false, true>(p, grid, v, nullptr, y, g, f, VecList{}, nullptr, out_scale);
    else
      stencil_fx_launch<kModeApply, 1>(p, grid, v, nullptr, y, g, f, VecList{}, nullptr, out_scale);
    BEC_LAUNCH_CHECK(p, "apply_L_fx_kernel");
    return BEC_OK;
  }
  BEC_LAUNCH_BEGIN(p);
#define BEC_L_LAUNCH(K, P)                                                \
  apply_L_kernel<K, P><<<stencil_grid(p), kStencilThreads, 0, p->stream>>>( \
      v, y, g, corner, out_scale)
  BEC_STENCIL_SWITCH(variant_of(p), BEC_L_LAUNCH)
#undef BEC_L_LAUNCH
  BEC_LAUNCH_CHECK(p, "apply_L_kernel");
  return BEC_OK;
}

bec_status launch_stencil_dots(bec_problem* p, const double* z, double* w,
                               const double* const* V, int nv, const double* sigma,
                               double* hout, const double* vshift, const double* sshift,
                               int norm_slot) {
  const bool fixed = fx_rows(p);
  const int most = fixed ? kFxDotVecs : kMaxVec, n = nv < most ? nv : most;
  VecList L;
  for (int i = 0; i < kMaxVec; ++i) L.v[i] = i < n ? V[i] : V[0];
  const int var = variant_of(p);
  const StencilGeom g = geom(p);
  int nb = kStencilDotBlocks;
  if (fixed) {
    FxStencil f;
    const unsigned grid = fx_stencil(p, g, f);
    nb = (int)grid;
    BEC_LAUNCH_BEGIN(p);
    switch (n) {
#define BEC_SFX_CASE(NV)                                                                    \
  case NV:                                                                                  \
    if (vshift == V[NV - 1])                                                                \
      stencil_fx_launch<kModeDots, NV, true>(p, grid, z, nullptr, w, g, f, L, vshift, sshift);  \
    else                                                                                    \
      stencil_fx_launch<kModeDots, NV>(p, grid, z, nullptr, w, g, f, L, vshift, sshift);    \
    break;
      BEC_SFX_CASE(1) BEC_SFX_CASE(2) BEC_SFX_CASE(3) BEC_SFX_CASE(4) BEC_SFX_CASE(5) BEC_SFX_CASE(6)
      BEC_SFX_CASE(7) BEC_SFX_CASE(8)
#undef BEC_SFX_CASE
      default: return BEC_EINVAL;
    }
    BEC_LAUNCH_CHECK(p, "stencil_dots_fx_kernel");
  } else {
    BEC_LAUNCH_BEGIN(p);
    switch (n) {
#define BEC_SD_CASE(NV)                                                                  \
    case NV:                                                                               \
      stencil_dots_launch<NV>(var, p->stream, z, w, g, L, vshift, sshift, p->partials);   \
      break;
      BEC_SD_CASE(1) BEC_SD_CASE(2) BEC_SD_CASE(3) BEC_SD_CASE(4) BEC_SD_CASE(5) BEC_SD_CASE(6)
      BEC_SD_CASE(7) BEC_SD_CASE(8) BEC_SD_CASE(9) BEC_SD_CASE(10) BEC_SD_CASE(11) BEC_SD_CASE(12)
      BEC_SD_CASE(13) BEC_SD_CASE(14) BEC_SD_CASE(15) BEC_SD_CASE(16) BEC_SD_CASE(17)
      BEC_SD_CASE(18) BEC_SD_CASE(19) BEC_SD_CASE(20) BEC_SD_CASE(21) BEC_SD_CASE(22)
      BEC_SD_CASE(23) BEC_SD_CASE(24) BEC_SD_CASE(25) BEC_SD_CASE(26) BEC_SD_CASE(27)
      BEC_SD_CASE(28) BEC_SD_CASE(29) BEC_SD_CASE(30) BEC_SD_CASE(31) BEC_SD_CASE(32)
#undef BEC_SD_CASE
      default: return BEC_EINVAL;
    }
    BEC_LAUNCH_CHECK(p, "stencil_dots_kernel");
  }
  const bec_status s = launch_finish_dots(p, n, nb, sigma, hout, nullptr, norm_slot);
  if (s != BEC_OK || nv <= most) return s;
  // more vectors than one fused launch holds: the rest as plain dots
  return launch_dots(p, w, V + most, nv - most, sigma ? sigma + most : nullptr, hout + most);
}

bec_status launch_residual(bec_problem* p, const double* f, const double* u, double* r) {
  const StencilGeom g = geom(p);
  if (u != nullptr && fx_rows(p)) {
    FxStencil x;
    const unsigned grid = fx_stencil(p, g, x);
    BEC_LAUNCH_BEGIN(p);
    stencil_fx_launch<kModeResidual, 1>(p, grid, u, f, r, g, x, VecList{}, nullptr, nullptr);
    BEC_LAUNCH_CHECK(p, "residual_fx_kernel");
    return BEC_OK;
  }
  BEC_LAUNCH_BEGIN(p);
#define BEC_R_LAUNCH(K, P) \
  residual_kernel<K, P><<<stencil_grid(p), kStencilThreads, 0, p->stream>>>(f, u, r, g)
  BEC_STENCIL_SWITCH(variant_of(p), BEC_R_LAUNCH)
#undef BEC_R_LAUNCH
  BEC_LAUNCH_CHECK(p, "residual_kernel");
  return BEC_OK;
}

bec_status launch_residual_norms(bec_problem* p, const double* f, const double* u, int slot, int fslot,
                                 bool to_host) {
  const dim3 grid = stencil_grid(p);
  const StencilGeom g = geom(p);
  long long nblk = (long long)grid.x * grid.y;
  if (fx_rows(p)) {
    FxStencil x;
    const unsigned gx = fx_stencil(p, g, x);
    nblk = gx;
    BEC_LAUNCH_BEGIN(p);
    if (fslot >= 0)
      stencil_fx_launch<kModeNorms, 1, true>(p, gx, u, f, nullptr, g, x, VecList{}, nullptr, nullptr);
    else
      stencil_fx_launch<kModeNorms, 1>(p, gx, u, f, nullptr, g, x, VecList{}, nullptr, nullptr);
    BEC_LAUNCH_CHECK(p, "residual_norms_fx_kernel");
  } else {
    BEC_LAUNCH_BEGIN(p);
#define BEC_RN_LAUNCH(K, P) \
    residual_norms_kernel<K, P><<<grid, kStencilThreads, 0, p->stream>>>(f, u, p->partials, g)
    BEC_STENCIL_SWITCH(variant_of(p), BEC_RN_LAUNCH)
#undef BEC_RN_LAUNCH
    BEC_LAUNCH_CHECK(p, "residual_norms_kernel");
  }
  BEC_LAUNCH_BEGIN(p);
  finish_norms_kernel<<<1, 256, 0, p->stream>>>(p->partials, nblk, p->scal, slot, fslot,
                                                to_host ? p->host_scal_dev : nullptr);
  BEC_LAUNCH_CHECK(p, "finish_norms_kernel");
  return BEC_OK;
}

bec_status launch_build_rhs(bec_problem* p, const double* u0, const double* fsrc, double* f) {
  BEC_LAUNCH_BEGIN(p);
  build_rhs_kernel<<<4 * 152, 256, 0, p->stream>>>(u0, fsrc, f, geom(p), p->tau);
  BEC_LAUNCH_CHECK(p, "build_rhs_kernel");
  return BEC_OK;
}

}  // namespace bec
