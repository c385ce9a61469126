// Per-element pieces of the forward step shared by the per-grid kernels and the
// batched ones: one domain-halo cell, one immersed-boundary ghost cell (Sec. 2, Fig. 1(c))
// and the CFL wave-speed rate of one cell.
#pragma once
#include <math_constants.h>
#include "js_device.cuh"
#include "js_internal.h"

namespace js {

// number of halo cells filled per grid: x sides on interior rows, y sides on the full width
__host__ __device__ __forceinline__ long long halo_count(const Lay& lay) {
  return 6LL * lay.ny + ((lay.ny > 1) ? 6LL * (lay.nx + 6) : 0);
}

// Fill halo cell number t (0 <= t < halo_count).  The y rule is resolved first (it reads
// x-ghost columns, which the x rule defines from interior cells), then the x rule;
// reflective sides flip the normal momentum, inflow sides hold a fixed state.
__device__ __forceinline__ void bc_fill_one(double* __restrict__ U, const Lay& lay, const BcArgs& bc, long long t) {
  const int nx = lay.nx, ny = lay.ny;
  const long long nxg = 6LL * ny;
  int di, dj;
  if (t < nxg) {
    dj = (int)(t / 6);
    const int r = (int)(t % 6);
    di = (r < 3) ? -(r + 1) : nx + (r - 3);
  } else {
    const long long u = t - nxg;
    di = (int)(u / 6) - 3;
    const int r = (int)(u % 6);
    dj = (r < 3) ? -(r + 1) : ny + (r - 3);
  }
  int i = di, j = dj;
  bool flipx = false, flipy = false;
  int side_inflow = -1;
  if (j < 0 || j >= ny) {
    const int side = (j < 0) ? 2 : 3;
    const int k = (j < 0) ? -j : j - ny + 1;
    switch (bc.kind[side]) {
      case 0: j = (side == 2) ? 0 : ny - 1; break;
      case 1: j = (side == 2) ? k - 1 : ny - k; flipy = true; break;
      case 2: j = (side == 2) ? ny - k : k - 1; break;
      default: side_inflow = side; break;
    }
  }
  if (side_inflow < 0 && (i < 0 || i >= nx)) {
    const int side = (i < 0) ? 0 : 1;
    const int k = (i < 0) ? -i : i - nx + 1;
    switch (bc.kind[side]) {
      case 0: i = (side == 0) ? 0 : nx - 1; break;
      case 1: i = (side == 0) ? k - 1 : nx - k; flipx = true; break;
      case 2: i = (side == 0) ? nx - k : k - 1; break;
      default: side_inflow = side; break;
    }
  }
  double v[4];
  if (side_inflow >= 0) {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = bc.inflow_cons[side_inflow][c];
  } else {
    const long long s = lay.idx(i, j);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = U[c * lay.plane + s];
  }
  if (flipx) v[1] = -v[1];
  if (flipy) v[2] = -v[2];
  const long long d = lay.idx(di, dj);
#pragma unroll
  for (int c = 0; c < 4; ++c) U[c * lay.plane + d] = v[c];
}

// sum over the four lanes of a quad (the same value on each: (0 + 1) + (2 + 3))
__device__ __forceinline__ double quad_sum(double x) {
  const unsigned m = 0xfu << (threadIdx.x & 28);
  x += __shfl_xor_sync(m, x, 1);
  return x + __shfl_xor_sync(m, x, 2);
}
__device__ __forceinline__ double pick4(int c, double a, double b, double d, double e) {
  return c < 2 ? (c == 0 ? a : b) : (c == 2 ? d : e);
}

// The image point of ghost cell k: primitives q = (rho, u, v, p) interpolated from its four source
// cells, lane m of the quad taking source m, and the velocity (ug, vg) mirrored at the wall.  A cell
// of weight 0 is not read.  Bound by latency: one load of weights and cells, one of states, one
// reciprocal, then sums over the quad.
__device__ __forceinline__ void ib_image(const double* __restrict__ U, const Lay& lay, const IbArgs& ib, double gm1,
                                         int wall, int k, int m, double q[4], double& nx, double& ny, double& ug,
                                         double& vg) {
  const double w = ib.w[4 * k + m];
  const long long s = ib.src[4 * k + m];
  nx = ib.nrm[2 * k];
  ny = ib.nrm[2 * k + 1];
  q[0] = q[1] = q[2] = q[3] = 0.0;
  if (w != 0.0) {
    const double r = U[s], mx = U[lay.plane + s], my = U[2 * lay.plane + s], E = U[3 * lay.plane + s];
    const u64 rr = recip_top(mant64(r));
    const double u = quot_near(mx, r, rr), v = quot_near(my, r, rr);
    q[0] = w * r;
    q[1] = w * u;
    q[2] = w * v;
    q[3] = w * (gm1 * (E - 0.5 * r * fma(u, u, v * v)));
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) q[c] = quad_sum(q[c]);
  if (wall == 0) {
    const double vn = fma(q[1], nx, q[2] * ny);
    ug = fma(-2.0 * vn, nx, q[1]);
    vg = fma(-2.0 * vn, ny, q[2]);
  } else {
    ug = -q[1];
    vg = -q[2];
  }
}

// Ghost cell t / 4, by lane t % 4 of a quad (t a multiple of 4 on the quad's first lane): slip-wall
// (or no-slip) mirror of the bilinear interpolation of fluid cells at its image point.
__device__ __forceinline__ void ib_fill_one(double* __restrict__ U, const Lay& lay, const IbArgs& ib, double gamma,
                                            int wall, int t) {
  const int k = t >> 2, m = t & 3;
  const double gm1 = gamma - 1.0;
  double q[4], nx, ny, ug, vg;
  const u64 rg = recip_top(mant64(gm1));
  ib_image(U, lay, ib, gm1, wall, k, m, q, nx, ny, ug, vg);
  const double e = fma(0.5 * q[0], fma(ug, ug, vg * vg), quot_near(q[3], gm1, rg));
  U[m * lay.plane + ib.dst[k]] = pick4(m, q[0], q[0] * ug, q[0] * vg, e);
}

// CFL rate (|u| + a)/dx [+ (|v| + a)/dy] of one cell with conserved values (r, mx, my, E),
// IEEE-rounded in the oracle's operation order.  A non-physical cell (rho or p not positive,
// or not finite) gets the rate +infinity: it dominates every maximum, so the step size of a
// state holding one is 0 and the CFL entry points report JS_ERR_NONPHYSICAL.
__device__ __forceinline__ double cfl_rate(double r, double mx, double my, double E, double gamma, double dx,
                                           double dy, bool two_d) {
  const double u = __ddiv_rn(mx, r), v = __ddiv_rn(my, r);
  const double ke = __dmul_rn(__dmul_rn(0.5, r), __dadd_rn(__dmul_rn(u, u), __dmul_rn(v, v)));
  const double p = __dmul_rn(gamma - 1.0, __dsub_rn(E, ke));
  if (!(r > 0.0) || !(r < CUDART_INF) || !(p > 0.0) || !(p < CUDART_INF)) return CUDART_INF;
  const double a = __dsqrt_rn(__ddiv_rn(__dmul_rn(gamma, p), r));
  double s = __ddiv_rn(__dadd_rn(fabs(u), a), dx);
  if (two_d) s = __dadd_rn(s, __ddiv_rn(__dadd_rn(fabs(v), a), dy));
  return s;
}

// The two-pass CFL reduction (js_forward.cu): rates within CFL_MARGIN/2 of cfl_rate's.
constexpr double CFL_MARGIN = 4e-5;

// in FP64 with the fast reciprocal where the approximation's error bound holds, else cfl_rate itself
__device__ __forceinline__ double cfl_rate_fast(double r, double mx, double my, double E, double gamma, double dx,
                                                double dy, double idx, double idy, bool two_d) {
  if (!(r > 1e-290) || !(r < 1e290)) return cfl_rate(r, mx, my, E, gamma, dx, dy, two_d);
  const double rr = recip(r);
  const double u = mx * rr, v = my * rr;
  const double ke = (0.5 * r) * fma(u, u, v * v);
  const double p = (gamma - 1.0) * (E - ke);
  // p <= 1e-8 E, p <= 0 or NaN: the approximation's error bound does not hold
  if (!(p > 1e-8 * E) || !(E < 1e290)) return cfl_rate(r, mx, my, E, gamma, dx, dy, two_d);
  const double c2 = (gamma * p) * rr;
  const double a = (c2 > 1e-290) ? c2 * rsqrt_nr(c2) : sqrt(c2);
  double s = (fabs(u) + a) * idx;
  if (two_d) s = fma(fabs(v) + a, idy, s);
  return s;
}

// In FP32: reading the doubles' upper bits costs integer instructions only, where FP64 arithmetic and
// conversions run at a fortieth of the FP32 rate.  Inputs truncated to 24 bits (relative 2^-23), the
// momentum quotient within 4 of those units, the kinetic energy within 11, so where E - ke > E/16 the
// pressure is within 16 * 12 + 2 and the sound speed within 100 units: 1.2e-5 < CFL_MARGIN/2.
struct CflF {
  float g, gm1, idx, idy;
  bool ok;  // the constants are in the range below
};
__device__ __forceinline__ bool mid_range(double x) {  // 2^-40 <= x < 2^40
  return (unsigned)(__double2hiint(x) - ((1023 - 40) << 20)) < (80u << 20);
}
// x truncated to a float, |x| < 2^100 (0 below 2^-100)
__device__ __forceinline__ float narrow(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x), m = h & 0x7fffffffu;
  const unsigned f = __funnelshift_l(l, m, 3) - (896u << 23);
  return __uint_as_float((h & 0x80000000u) | (m < ((1023u - 100u) << 20) ? 0u : f));
}
__device__ __forceinline__ CflF cfl_f32(double gamma, double idx, double idy, bool two_d) {
  const double gm1 = gamma - 1.0;
  if (!two_d) idy = 1.0;
  return CflF{narrow(gamma), narrow(gm1), narrow(idx), narrow(idy),
              gm1 > 1e-3 && gamma < 1e3 && mid_range(idx) && mid_range(idy)};
}
// false: not within the bound (s unset)
__device__ __forceinline__ bool cfl_rate_f32(double r, double mx, double my, double E, const CflF& c, bool two_d,
                                             float& s) {
  constexpr unsigned M = (1023u + 100u) << 20;
  if (!(c.ok && mid_range(r) && mid_range(E) && ((unsigned)__double2hiint(mx) & 0x7fffffffu) < M &&
        ((unsigned)__double2hiint(my) & 0x7fffffffu) < M))
    return false;
  const float rf = narrow(r), ef = narrow(E), rr = __fdividef(1.0f, rf);
  const float u = narrow(mx) * rr, v = narrow(my) * rr;
  const float ei = fmaf(-0.5f * rf, fmaf(u, u, v * v), ef);
  if (!(ei > 0.0625f * ef)) return false;
  const float c2 = c.g * (c.gm1 * ei) * rr;
  const float a = c2 * rsqrtf(c2);
  s = (fabsf(u) + a) * c.idx;
  if (two_d) s = fmaf(fabsf(v) + a, c.idy, s);
  return true;
}
// one cell's approximate rate into the running maxima rf, rd (their larger one counts)
__device__ __forceinline__ void cfl_rate_max(double r, double mx, double my, double E, double gamma, double dx,
                                             double dy, double idx, double idy, const CflF& c, bool two_d, float& rf,
                                             double& rd) {
  float s;
  if (cfl_rate_f32(r, mx, my, E, c, two_d, s)) rf = fmaxf(rf, s);
  else rd = fmax(rd, cfl_rate_fast(r, mx, my, E, gamma, dx, dy, idx, idy, two_d));
}
// whether that rate reaches thr
__device__ __forceinline__ bool cfl_reaches(double r, double mx, double my, double E, double gamma, double dx,
                                            double dy, double idx, double idy, const CflF& c, bool two_d, double thr) {
  float s;
  if (cfl_rate_f32(r, mx, my, E, c, two_d, s)) return (double)s >= thr;
  return cfl_rate_fast(r, mx, my, E, gamma, dx, dy, idx, idy, two_d) >= thr;
}

// bitwise equality of two states (identical states have identical IEEE rates)
__device__ __forceinline__ bool same_bits(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}

}  // namespace js
