// Device bodies of the reverse-mode stage (gradient chain rule of Sec. 2 applied to the
// discrete operator), shared by the per-grid launches of js_adjoint.cu and the persistent
// batched reverse kernel of js_batch.cu: one tile, element or block of each phase.
#pragma once
#include <cuda_runtime.h>

#include "js_adjoint_device.cuh"
#include "js_internal.h"

namespace js {

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Per-warp partial sums of the parameter gradient's gamma, mu, Pr and nu entries:
// pp[4 * w + k] = the sum over warp w's lanes (a fixed shuffle tree), w = the warp's global
// index (thread index / 32 over the launch).  Every lane calls it (no lane may have left);
// pp == nullptr (no pbar) skips it.  The partials are summed in warp order at the end of the
// stage, so the parameter gradient does not depend on timing, and two launch shapes that map
// the same items to the same warps give the same bits.
__device__ __forceinline__ void warp_partials(double* pp, long long w, double g, double m, double pr, double n) {
  if (pp == nullptr) return;
  g = warp_sum(g);
  m = warp_sum(m);
  pr = warp_sum(pr);
  n = warp_sum(n);
  if ((threadIdx.x & 31) == 0) {
    double* o = pp + 4 * w;
    o[0] = g;
    o[1] = m;
    o[2] = pr;
    o[3] = n;
  }
}
__device__ __forceinline__ long long global_warp() {
  return ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}

// Position of face k of line `line` in the planes of the neural flux's face-state adjoints: y lines
// use the padded layout, x lines are stored transposed (its kernel runs lanes across the lines in
// both directions).
__device__ __forceinline__ long long face_id(const AdjArgs& a, int dir, int k, int line) {
  return dir == 0 ? (long long)(k + 3) * a.tpitch + (line + a.lay.gy) : a.lay.idx(line, k);
}

// =======================================================================================
// Reverse of one stage on one tile of the padded array: given the adjoint Unext of the stage
// output and the filled stage state X,
//   lambda' = b dt Unext on fluid cells (0 elsewhere), U^n part Uacc += a Unext,
//   Ub(X) = identity and carry terms + (dprim/dX)^T (reverse of the x and y fluxes) + nu lap(lambda')
// in one pass: primitives and lambda' of the tile and its halo in shared memory, then per line
// (a warp each, a lane per cell, as in the stage kernel) WENO5 forward, HLLC and viscous forward and
// reverse per face, WENO5 reverse.  Of the 32 cells of lanes 0..31 the differences serve WENO5 of
// lanes 1..30, these the faces at i+1/2 of lanes 1..29, these the WENO5 reverse of lanes 2..29 and
// these the primitive adjoints of lanes 4..27: the 24 outputs.  Nothing is stored between: the
// WENO5 internals, face adjoints and segment sums that separate passes kept in memory (1.3 KB a
// cell) are recomputed in integer arithmetic beside the FP64 pipe or passed by shuffles.
// Every sum has a fixed order, so the reverse pass gives the same bits on every run.
// =======================================================================================
constexpr int AB = 34;              // box of the tile: outputs at 5 .. 28
constexpr int AP = AB * AB;
constexpr int AQ = ADJ_TILE + 1;    // row pitch of the accumulator planes
constexpr int AA = ADJ_TILE * AQ;
constexpr int AS = (ADJ_TILE + 2) * AQ;  // tangential terms: lines -1 .. 24
// doubles of shared memory: 4 planes of primitives, 4 of lambda', accumulators (5 viscous), 2 planes
// of tangential terms (viscous)
template <bool VISC>
__host__ __device__ constexpr size_t adj_smem() {
  return sizeof(double) * (size_t)(8 * AP + (VISC ? 5 * AA + 2 * AS : 4 * AA));
}

// the reverse of one line at the lane's cell (q: primitives, l: lambda'; neighbours at multiples of
// st, across the line of ts).  f: number of the face at i+1/2 (faces 0 .. n exist), own: the lane's
// face counts for the parameter gradient, out(c, v) receives the adjoint of primitive c (lanes
// 4..27), tang(n, t) the cell's tangential terms of its two faces (VISC, 2D).
template <bool VISC, bool HAS_T, class Nn, class Out, class Tang>
__device__ __forceinline__ void adj_line(const double* q, const double* l, int st, int ts, int pn, int f, int n,
                                         const Gas& g, const ViscC& vc, double invh, bool own, double& gs1,
                                         double& gs2, double& vmu, double& vk, Nn nn, Out out, Tang tang) {
  const int lane = threadIdx.x & 31;
  const bool inner = lane - 1u < 30u;
  const int pt = 3 - pn;
  const bool face = lane >= 1 && lane <= 29 && f >= 0 && f <= n;
  double L[4], R[4];
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    const int c = (k == 1) ? pn : (k == 2) ? pt : k;
    double Lf, Rf;
    weno_lane(q + c * AP, st, k == 0 || k == 3, inner, Lf, Rf);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      L[m] = (k == m) ? Lf : L[m];
      R[m] = (k == m) ? Rf : R[m];
    }
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) R[m] = __shfl_down_sync(0xffffffffu, R[m], 1);
  const double* un = q + pn * AP;
  const double* ut = q + pt * AP;
  const bool fallback = !(positive(L[0]) && positive(L[3]) && positive(R[0]) && positive(R[3]));
  if (fallback) {
    L[0] = q[0], L[1] = un[0], L[2] = ut[0], L[3] = q[3 * AP];
    R[0] = q[st], R[1] = un[st], R[2] = ut[st], R[3] = q[3 * AP + st];
  }
  double Fb[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    const double* lm = l + (m == 1 ? pn : m == 2 ? pt : m) * AP;
    Fb[m] = (lm[st] - lm[0]) * invh;
  }
  double bL[4], bR[4], s1 = 0.0, s2 = 0.0;
  hllc_vjp(L, R, g, Fb, bL, bR, s1, s2);
  if (own && face) {
    gs1 += s1;
    gs2 += s2;
  }
  // adjoints that go straight to the face's cells: its left cell (dl) and its right cell (dr)
  double dl[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, dr[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    dl[m] = fallback && face ? bL[m] : 0.0;
    dr[m] = fallback && face ? bR[m] : 0.0;
    bL[m] = fallback || !face ? 0.0 : bL[m];
    bR[m] = fallback || !face ? 0.0 : bR[m];
  }
  nn(face, bL, bR);
  bool straight = __any_sync(0xffffffffu, fallback && face);
  if (VISC) {
    // F[n] -= tnn; F[t] -= tnt; F[3] -= 0.5 (sbn tnn + sbt tnt) + ck dT
    const double Tc = q[3 * AP] * recip(q[0]);
    const double dT = __shfl_down_sync(0xffffffffu, Tc, 1) - Tc;
    const double ua = un[0], ub = un[st], ta = ut[0], tb = ut[st];
    const double dun = ub - ua, dut = tb - ta;
    double tnn, tnt;
    if (HAS_T) {
      const double sun = (un[ts] - un[-ts]) + (un[st + ts] - un[st - ts]);
      const double sut = (ut[ts] - ut[-ts]) + (ut[st + ts] - ut[st - ts]);
      tnn = fma(vc.c43n, dun, -vc.c23t * sut);
      tnt = fma(vc.cn, dut, vc.ct * sun);
    } else {
      tnn = vc.c43n * dun;
      tnt = vc.cn * dut;
    }
    const double h3 = 0.5 * Fb[3];
    const double btnn = fma(-h3, ua + ub, -Fb[1]), btnt = fma(-h3, ta + tb, -Fb[2]);
    const double bck = -Fb[3] * dT, bdT = -Fb[3] * vc.ck;
    const double bn = -h3 * tnn, bt = -h3 * tnt, bdun = vc.c43n * btnn, bdut = vc.cn * btnt;
    if (face) {
      dl[1] += bn - bdun;
      dr[1] += bn + bdun;
      dl[2] += bt - bdut;
      dr[2] += bt + bdut;
      dl[4] = -bdT;
      dr[4] = bdT;
      if (own) {
        vmu += fma(btnn, tnn, fma(btnt, tnt, bck * vc.ck));
        vk += bck * vc.ck;
      }
    }
    if (HAS_T) {
      // tangential differences: + to the cells one line up, minus to those one line down
      const double xn = face ? vc.ct * btnt : 0.0, xt = face ? -vc.c23t * btnn : 0.0;
      tang(xn + __shfl_up_sync(0xffffffffu, xn, 1), xt + __shfl_up_sync(0xffffffffu, xt, 1));
    }
    straight = true;
  }
  if (straight) {
#pragma unroll
    for (int m = 0; m < (VISC ? 5 : 4); ++m)
      out((m == 1) ? pn : (m == 2) ? pt : m, dl[m] + __shfl_up_sync(0xffffffffu, dr[m], 1));
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) bR[m] = __shfl_up_sync(0xffffffffu, bR[m], 1);  // of the face at i-1/2
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    const int c = (k == 1) ? pn : (k == 2) ? pt : k;
    const double Lb = (k == 0) ? bL[0] : (k == 1) ? bL[1] : (k == 2) ? bL[2] : bL[3];
    const double Rb = (k == 0) ? bR[0] : (k == 1) ? bR[1] : (k == 2) ? bR[2] : bR[3];
    double w[4];
    weno_grad_lane(q + c * AP, st, k == 0 || k == 3, inner, Lb, Rb, w);
    // adjoint of d_{i+1/2}: its share in the cells i-1 .. i+2
    const double t = (w[2] + __shfl_up_sync(0xffffffffu, w[3], 1)) +
                     (__shfl_down_sync(0xffffffffu, w[1], 1) + __shfl_down_sync(0xffffffffu, w[0], 2));
    out(c, fma(SIXTH, __shfl_up_sync(0xffffffffu, t, 1) - t, Lb + Rb));
  }
}

// tile (bx, by) of the padded array; slot0: warp slot of the tile's partials of pbar[0..3]
template <bool VISC>
__device__ __forceinline__ void adj_tile(const AdjArgs& a, const double* __restrict__ Unext, double* __restrict__ Uacc,
                                         double ra, double rb, double dt, int rhs_mode, int bx, int by, double* smem,
                                         long long slot0) {
  const Lay& L = a.lay;
  double* sq = smem;
  double* sl = smem + 4 * AP;
  double* acc = smem + 8 * AP;
  double* tan = acc + 5 * AA;  // VISC
  const Gas g = a.gas;
  const int W = L.nx + 6;
  const int ox = bx * ADJ_TILE, oy = by * ADJ_TILE;  // padded coordinates of the first output
  const double bdt = rhs_mode ? 1.0 : rb * dt;
  for (int e = threadIdx.x; e < AP; e += blockDim.x) {
    const int row = e / AB, col = e - row * AB;
    const int gx = ox - 5 + col, gy = oy - 5 + row;
    const bool in = gx >= 0 && gx < W && gy >= 0 && gy < L.H;
    const long long t = in ? (long long)gy * L.pitch + gx : 0;
    const double r = a.X[t], mx = a.X[L.plane + t], my = a.X[2 * L.plane + t], E = a.X[3 * L.plane + t];
    double u = 0.0, v = 0.0, p = 1.0, T;
    if (in) cons_to_prim(r, mx, my, E, g, u, v, p, T);
    sq[e] = in ? r : 1.0;
    sq[AP + e] = u;
    sq[2 * AP + e] = v;
    sq[3 * AP + e] = p;
    const int i = gx - 3, j = gy - L.gy;
    const bool fluid = i >= 0 && i < L.nx && j >= 0 && j < L.ny && (a.tag == nullptr || a.tag[(long long)j * L.nx + i] == 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) sl[c * AP + e] = fluid ? bdt * Unext[c * L.plane + t] : 0.0;
  }
  for (int e = threadIdx.x; e < (VISC ? 5 : 4) * AA; e += blockDim.x) acc[e] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int k = lane - 4;  // the lane's cell: output k of the line
  const bool own = k >= 0 && k < ADJ_TILE;
  double gs1 = 0.0, gs2 = 0.0, vmu = 0.0, vk = 0.0, gb = 0.0, nb = 0.0;
#pragma unroll 1
  for (int dir = 0; dir < (a.two_d ? 2 : 1); ++dir) {
    const int st = dir == 0 ? 1 : AB, ts = dir == 0 ? AB : 1;
    const int k0 = (dir == 0 ? ox - 3 : oy - L.gy), l0 = (dir == 0 ? oy - L.gy : ox - 3);  // grid cell of output 0
    const int nline = dir == 0 ? L.ny : L.nx, ncell = dir == 0 ? L.nx : L.ny;
    const ViscC vc = dir == 0 ? a.vx : a.vy;
    const double invh = dir == 0 ? a.inv_dx : a.inv_dy;
    const int pn = dir + 1;
    // with tangential terms the lines next to the tile are needed for those alone
    const int edge = VISC && a.two_d ? 1 : 0;
#pragma unroll 1
    for (int ln = warp - edge; ln < ADJ_TILE + edge; ln += nwarp) {
      const double* q = sq + (ln + 5) * ts + (k + 5) * st;
      const double* lm = sl + (ln + 5) * ts + (k + 5) * st;
      const int line = l0 + ln, f = k0 + k + 1;
      if (VISC && a.two_d && (ln < 0 || ln >= ADJ_TILE || line < 0 || line >= nline)) {
        // tangential terms only (zero past the grid's lines)
        double xn = 0.0, xt = 0.0;
        if (line >= 0 && line < nline && lane >= 1 && lane <= 29 && f >= 0 && f <= ncell) {
          const double* un = q + pn * AP;
          const double* ut = q + (3 - pn) * AP;
          const double h3 = 0.5 * ((lm[3 * AP + st] - lm[3 * AP]) * invh);
          const double Fn = (lm[pn * AP + st] - lm[pn * AP]) * invh, Ft = (lm[(3 - pn) * AP + st] - lm[(3 - pn) * AP]) * invh;
          xn = vc.ct * fma(-h3, ut[0] + ut[st], -Ft);
          xt = -vc.c23t * fma(-h3, un[0] + un[st], -Fn);
        }
        const double xn1 = __shfl_up_sync(0xffffffffu, xn, 1), xt1 = __shfl_up_sync(0xffffffffu, xt, 1);
        if (own) {
          tan[(ln + 1) * AQ + k] = xn + xn1;
          tan[AS + (ln + 1) * AQ + k] = xt + xt1;
        }
        continue;
      }
      if (line < 0 || line >= nline) continue;
      double* o = acc + (dir == 0 ? ln * AQ + k : k * AQ + ln);
      auto nn = [&](bool face, double bL[4], double bR[4]) {
        if (a.fadj == nullptr || !face) return;
        const long long si = face_id(a, dir, f, line);
        const double* fa = a.fadj + (long long)(dir * 8) * a.splane + si;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int c = (m == 1) ? pn : (m == 2) ? 3 - pn : m;
          bL[m] += fa[c * a.splane];
          bR[m] += fa[(4 + c) * a.splane];
        }
      };
      auto out = [&](int c, double v) {
        if (own) o[c * AA] += v;
      };
      auto tang = [&](double xn, double xt) {
        if (own) {
          tan[(ln + 1) * AQ + k] = xn;
          tan[AS + (ln + 1) * AQ + k] = xt;
        }
      };
      if (a.two_d) adj_line<VISC, true>(q, lm, st, ts, pn, f, ncell, g, vc, invh, own, gs1, gs2, vmu, vk, nn, out, tang);
      else adj_line<VISC, false>(q, lm, st, ts, pn, f, ncell, g, vc, invh, own, gs1, gs2, vmu, vk, nn, out, tang);
    }
    __syncthreads();
    if (VISC && a.two_d) {
      // tangential terms: from the line below and, negative, from the line above
      for (int e = threadIdx.x; e < ADJ_TILE * ADJ_TILE; e += blockDim.x) {
        const int ln = e / ADJ_TILE, kk = e - ln * ADJ_TILE;
        double* o = acc + (dir == 0 ? ln * AQ + kk : kk * AQ + ln);
        o[pn * AA] += tan[ln * AQ + kk] - tan[(ln + 2) * AQ + kk];
        o[(3 - pn) * AA] += tan[AS + ln * AQ + kk] - tan[AS + (ln + 2) * AQ + kk];
      }
      __syncthreads();
    }
  }
  // primitive reverse, artificial viscosity, identity terms
  for (int e = threadIdx.x; e < ADJ_TILE * ADJ_TILE; e += blockDim.x) {
    const int ty = e / ADJ_TILE, tx = e - ty * ADJ_TILE;
    const int gx = ox + tx, gy = oy + ty;
    if (gx >= W || gy >= L.H) continue;
    const int i = gx - 3, j = gy - L.gy;
    const long long t = (long long)gy * L.pitch + gx;
    const int b = (ty + 5) * AB + tx + 5;
    double qb[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, ub[4];
#pragma unroll
    for (int c = 0; c < (VISC ? 5 : 4); ++c) qb[c] = acc[c * AA + ty * AQ + tx];
    prim_vjp(sq[b], sq[AP + b], sq[2 * AP + b], sq[3 * AP + b], g, qb, ub, gb);
    const bool interior = i >= 0 && i < L.nx && j >= 0 && j < L.ny;
    if (a.has_av) {
      const bool near = i >= -1 && i <= L.nx && j >= (a.two_d ? -1 : 0) && j <= (a.two_d ? L.ny : 0);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double* lam = sl + c * AP + b;
        if (near) {
          double add = a.nu_x * ((lam[-1] - 2.0 * lam[0]) + lam[1]);
          if (a.two_d) add += a.nu_y * ((lam[-AB] - 2.0 * lam[0]) + lam[AB]);
          ub[c] += add;
        }
        if (interior && lam[0] != 0.0) {
          const double* X = a.X + c * L.plane;
          double lap = a.nu_x1 * ((X[t - 1] - 2.0 * X[t]) + X[t + 1]);
          if (a.two_d) lap += a.nu_y1 * ((X[t - L.pitch] - 2.0 * X[t]) + X[t + L.pitch]);
          nb += lam[0] * lap;
        }
      }
    }
    const bool fluid = interior && (a.tag == nullptr || a.tag[(long long)j * L.nx + i] == 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const long long o = c * L.plane + t;
      if (interior && !rhs_mode) {
        const double un = Unext[o];
        ub[c] += fluid ? rb * un : un;  // identity on fluid cells, carry on solid and ghost cells
        if (fluid && ra != 0.0) Uacc[o] += ra * un;
      }
      a.Ub[o] = ub[c];
    }
  }
  gb += gs2 / g.gamma - gs1 * g.g1 * g.g1;
  if (VISC) {
    gb += a.kg * vk;
    vmu *= a.inv_mu;
    vk *= a.kp;
  }
  warp_partials(a.pp, slot0 + warp, gb, vmu, vk, nb);
}

// =======================================================================================
// transposed halo fill (gathers).  y sides first: targets are cells of interior rows (all
// padded columns); then x sides: targets are interior cells.
// =======================================================================================
__device__ __forceinline__ bool halo_source(int kind, int k, int n, bool low, int& src, bool& flip) {
  flip = false;
  switch (kind) {
    case 0: src = low ? 0 : n - 1; return true;
    case 1: src = low ? k - 1 : n - k; flip = true; return true;
    case 2: src = low ? n - k : k - 1; return true;
    default: return false;  // inflow
  }
}

__device__ __forceinline__ void adj_bcT_one(const AdjArgs& a, const BcArgs& bc, int phase_y, double* inflow_part,
                                            int tmax, long long t) {
  const Lay& L = a.lay;
  // targets: 6 source rows/columns next to each boundary
  const int ntan = phase_y ? L.nx + 6 : L.ny;
  if (t < 6LL * ntan) {
    const int r = (int)(t % 6);
    const int tan = (int)(t / 6) - (phase_y ? 3 : 0);
    const int n = phase_y ? L.ny : L.nx;
    const int tgt = (r < 3) ? r : n - 6 + r;  // 0,1,2, n-3,n-2,n-1
    const int comp = phase_y ? 2 : 1;          // momentum component normal to the side
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int s = 0; s < 2; ++s) {
      const int side = (phase_y ? 2 : 0) + s;
      for (int k = 1; k <= 3; ++k) {
        int src;
        bool flip;
        if (!halo_source(bc.kind[side], k, n, s == 0, src, flip) || src != tgt) continue;
        const int h = (s == 0) ? -k : n - 1 + k;
        const long long hid = phase_y ? L.idx(tan, h) : L.idx(h, tan);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const double v = a.Ub[c * L.plane + hid];
          acc[c] += (flip && c == comp) ? -v : v;
        }
      }
    }
    const long long tid = phase_y ? L.idx(tan, tgt) : L.idx(tgt, tan);
#pragma unroll
    for (int c = 0; c < 4; ++c) a.Ub[c * L.plane + tid] += acc[c];
  }
  // inflow sides: the halo adjoints of each (side, tangential position), its three layers in
  // order, into inflow_part[side][position] (summed over positions by adj_inflow_kernel)
  if (t < 2LL * ntan) {
    const int s = (int)(t % 2);
    const int tpos = (int)(t / 2);  // 0 .. ntan - 1
    const int tan = tpos - (phase_y ? 3 : 0);
    const int side = (phase_y ? 2 : 0) + s;
    if (bc.kind[side] == 3) {
      const int n = phase_y ? L.ny : L.nx;
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      for (int k = 1; k <= 3; ++k) {
        const int h = (s == 0) ? -k : n - 1 + k;
        const long long hid = phase_y ? L.idx(tan, h) : L.idx(h, tan);
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] += a.Ub[c * L.plane + hid];
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) inflow_part[((long long)side * tmax + tpos) * 4 + c] = acc[c];
    }
  }
}

// inflow halo adjoints (conserved) -> gradient of the inflow primitive state and gamma; one
// warp per side sums its partials in a fixed order, then one thread adds to pbar side by side
__device__ __forceinline__ void adj_inflow_block(const AdjArgs& a, const BcArgs& bc, const double* inflow_part,
                                                 int tmax, const double* inflow_prim) {
  __shared__ double S[4][4];
  const int side = threadIdx.x >> 5, lane = threadIdx.x & 31;  // (at least four warps)
  const Lay& L = a.lay;
  if (side < 4 && bc.kind[side] == 3 && a.pbar != nullptr) {
    const int ntan = (side < 2) ? L.ny : L.nx + 6;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = lane; k < ntan; k += 32)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] += inflow_part[((long long)side * tmax + k) * 4 + c];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = warp_sum(v[c]);
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < 4; ++c) S[side][c] = v[c];
  }
  __syncthreads();
  if (threadIdx.x != 0 || a.pbar == nullptr) return;
  for (int sd = 0; sd < 4; ++sd) {
    if (bc.kind[sd] != 3) continue;
    const double* s = S[sd];
    const double r = inflow_prim[4 * sd], u = inflow_prim[4 * sd + 1], v = inflow_prim[4 * sd + 2],
                 p = inflow_prim[4 * sd + 3];
    // U = (r, r u, r v, p/(gamma-1) + r (u^2 + v^2)/2)
    a.pbar[4 + 4 * sd + 0] += s[0] + s[1] * u + s[2] * v + s[3] * 0.5 * (u * u + v * v);
    a.pbar[4 + 4 * sd + 1] += s[1] * r + s[3] * r * u;
    a.pbar[4 + 4 * sd + 2] += s[2] * r + s[3] * r * v;
    a.pbar[4 + 4 * sd + 3] += s[3] * a.gas.g1;
    a.pbar[0] += -s[3] * p * a.gas.g1 * a.gas.g1;
  }
}

// pbar[0..3] += the warp partials pp[4 * b + k] of the slot ranges [off[r], off[r] + cnt[r]),
// r < nr: each thread over a fixed set of slots, then a fixed reduction tree over the block
// (blockDim.x a power of two, at most 256)
__device__ __forceinline__ void adj_pbar_reduce_block(const double* __restrict__ pp, const long long* off,
                                                      const long long* cnt, int nr, double* pbar) {
  __shared__ double red[4][256];
  const int nt = blockDim.x;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int r = 0; r < nr; ++r)
    for (long long b = threadIdx.x; b < cnt[r]; b += nt)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] += pp[4 * (off[r] + b) + k];
#pragma unroll
  for (int k = 0; k < 4; ++k) red[k][threadIdx.x] = v[k];
  __syncthreads();
  for (int w = nt / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < 4; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 4) pbar[threadIdx.x] += red[threadIdx.x][0];
  __syncthreads();
}

// =======================================================================================
// transposed immersed-boundary fill
// =======================================================================================
__device__ __forceinline__ void adj_ib_ghost_one(const AdjArgs& a, const IbArgs& ib, int wall, double* qIb, int k,
                                                 double& gb) {
  if (k < ib.n) {
    const Lay& L = a.lay;
    const double gamma = a.gas.gamma;
    double q[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const double w = ib.w[4 * k + m];
      if (w == 0.0) continue;
      const long long s = ib.src[4 * k + m];
      const double r = a.X[s], u = a.X[L.plane + s] / r, v = a.X[2 * L.plane + s] / r;
      const double p = (gamma - 1.0) * (a.X[3 * L.plane + s] - 0.5 * r * (u * u + v * v));
      q[0] += w * r;
      q[1] += w * u;
      q[2] += w * v;
      q[3] += w * p;
    }
    const double nx = ib.nrm[2 * k], ny = ib.nrm[2 * k + 1];
    double ug, vg;
    if (wall == 0) {
      const double vn = q[1] * nx + q[2] * ny;
      ug = q[1] - 2.0 * vn * nx;
      vg = q[2] - 2.0 * vn * ny;
    } else {
      ug = -q[1];
      vg = -q[2];
    }
    const long long d = ib.dst[k];
    double G[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      G[c] = a.Ub[c * L.plane + d];
      a.Ub[c * L.plane + d] = 0.0;  // the ghost's own input value is overwritten by the fill
    }
    // G = (r, r ug, r vg, p/(gamma-1) + r (ug^2 + vg^2)/2)
    const double br = G[0] + G[1] * ug + G[2] * vg + G[3] * 0.5 * (ug * ug + vg * vg);
    const double bug = G[1] * q[0] + G[3] * q[0] * ug;
    const double bvg = G[2] * q[0] + G[3] * q[0] * vg;
    const double g1 = a.gas.g1;
    gb -= G[3] * q[3] * g1 * g1;
    double bu, bv;
    if (wall == 0) {  // (ug, vg) = (I - 2 n n^T)(u, v): symmetric
      const double bn = bug * nx + bvg * ny;
      bu = bug - 2.0 * bn * nx;
      bv = bvg - 2.0 * bn * ny;
    } else {
      bu = -bug;
      bv = -bvg;
    }
    qIb[4 * k] = br;
    qIb[4 * k + 1] = bu;
    qIb[4 * k + 2] = bv;
    qIb[4 * k + 3] = G[3] * g1;
  }
}

__device__ __forceinline__ void adj_ib_src_one(const AdjArgs& a, const IbTArgs& tb, const double* qIb, int s,
                                               double& gb) {
  if (s < tb.nsrc) {
    double S[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int e = tb.ptr[s]; e < tb.ptr[s + 1]; ++e) {
      const int k = tb.ghost[e];
      const double w = tb.w[e];
#pragma unroll
      for (int c = 0; c < 4; ++c) S[c] += w * qIb[4 * k + c];
    }
    const Lay& L = a.lay;
    const long long id = tb.cell[s];
    // the fill used IEEE-rounded primitives; their derivative is the same map
    double ub[4];
    double u, v, p, T;
    const double r = a.X[id];
    cons_to_prim(r, a.X[L.plane + id], a.X[2 * L.plane + id], a.X[3 * L.plane + id], a.gas, u, v, p, T);
    prim_vjp(r, u, v, p, a.gas, S, ub, gb);
#pragma unroll
    for (int c = 0; c < 4; ++c) a.Ub[c * L.plane + id] += ub[c];
  }
}

// =======================================================================================
// small elementwise helpers
// =======================================================================================
__device__ __forceinline__ void adj_unpack_add_one(const double* __restrict__ P, const double* __restrict__ P2,
                                                   double* __restrict__ U, const Lay& lay, long long t) {
  const long long n = (long long)lay.nx * lay.ny;
  if (t >= 4 * n) return;
  const int c = (int)(t / n);
  const long long o = t % n;
  const int i = (int)(o % lay.nx), j = (int)(o / lay.nx);
  const long long id = c * lay.plane + lay.idx(i, j);
  U[t] = P2 ? P[id] + P2[id] : P[id];
}

}  // namespace js
