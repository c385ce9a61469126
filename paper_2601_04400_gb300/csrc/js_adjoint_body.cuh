// Device bodies of the reverse-mode stage (gradient chain rule of Sec. 2 applied to the
// discrete operator), shared by the per-grid launches of js_adjoint.cu and the
// batched ones of js_batch.cu: one element or block of each phase.
#pragma once
#include <cuda_runtime.h>

#include "js_adjoint_device.cuh"
#include "js_fill.cuh"
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
//
// The four sums of a warp by halves: lane l ends with the sum over all lanes of value l / 8.  Six
// FP64 additions where four trees take twenty.
__device__ __forceinline__ double warp_sum4(double a, double b, double c, double d) {
  const unsigned full = 0xffffffffu;
  const bool h = threadIdx.x & 16, q = threadIdx.x & 8;
  const double x = (h ? c : a) + __shfl_xor_sync(full, h ? a : c, 16);
  const double y = (h ? d : b) + __shfl_xor_sync(full, h ? b : d, 16);
  double v = (q ? y : x) + __shfl_xor_sync(full, q ? x : y, 8);
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
  return v;
}
__device__ __forceinline__ void warp_partials(double* pp, long long w, double g, double m, double pr, double n) {
  if (pp == nullptr) return;
  const double v = warp_sum4(g, m, pr, n);
  if ((threadIdx.x & 7) == 0) pp[4 * w + ((threadIdx.x & 31) >> 3)] = v;
}
// the block's sums of the four values over its warps in order (at most 8 warps, all threads call it): value
// k on thread k < 4, 0 on the others
__device__ __forceinline__ double block_sum4(double a, double b, double c, double d) {
  __shared__ double part[8][4];
  const double v = warp_sum4(a, b, c, d);
  if ((threadIdx.x & 7) == 0) part[threadIdx.x >> 5][(threadIdx.x & 31) >> 3] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 4)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w][threadIdx.x];
  return t;
}
// the same into one slot a block, so that the final reduction stays short
__device__ __forceinline__ void block_partials(double* pp, long long slot, double g, double m, double pr, double n) {
  if (pp == nullptr) return;
  const double t = block_sum4(g, m, pr, n);
  if (threadIdx.x < 4) pp[4 * slot + threadIdx.x] = t;
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
// Reverse of one stage, given the adjoint Unext of the stage output and the filled stage state X:
//   lambda' = b dt Unext on fluid cells (0 elsewhere), U^n part Uacc += a Unext,
//   Ub(X) = identity and carry terms + (dprim/dX)^T (reverse of the x and y fluxes) + nu lap(lambda')
// in two launches: lines (the reverse of the fluxes of every x and y line, to primitive adjoints in
// memory) and cells (their sum through the primitive map).
//
// A warp takes 28 cells of one line, a lane one cell, as in the stage kernel: WENO5 forward, HLLC
// and viscous forward and reverse per face, WENO5 reverse.  Lanes 0..31 hold the cells i0 - 2 ..
// i0 + 29; the differences serve WENO5 of lanes 1..30, these the faces at i+1/2 of lanes 1..29,
// these the WENO5 reverse of lanes 2..29, whose 28 cells send primitive adjoints to all 32: those of
// the outer two on either side go to strips that the cell launch adds to the neighbouring warps'
// sums.  28 of 32 lanes' work is kept (24 when a warp formed complete sums alone).
// Nothing else is stored between forward and reverse: the WENO5 internals, face adjoints and segment
// sums that separate passes kept in memory (1.3 KB a cell) are recomputed in integer arithmetic
// beside the FP64 pipe or passed by shuffles.  Lines are independent, so that a grid of a few
// thousand lines fills the GPU (a 24x24-tile kernel of the same arithmetic took 234 us a stage at
// 250x190, six lines in turn per warp).
// Every sum has a fixed order, so the reverse pass gives the same bits on every run.
// =======================================================================================
constexpr int AB = 34;                   // positions of a line's box: lane l at l + 1
constexpr int ADJ_SPLIT = ADJ_LINES / 4;  // lines a block where four warps share one
// plane of a block's box, [line][position] in both directions: nl lines and one on either side
__host__ __device__ constexpr int adj_plane(int nl) { return AB * (nl + 2); }
// shared doubles of a block: the box's 8 planes; shared lines: 12 rows of a warp's lanes a line
__host__ __device__ constexpr int adj_smem(bool split) {
  return 8 * adj_plane(split ? ADJ_SPLIT : ADJ_LINES) + (split ? ADJ_SPLIT * 12 * 32 : 0);
}
// line blocks of a direction: groups of ADJ_LINES lines x chunks of 28 cells (-1 .. n) along them
__host__ __device__ inline int adj_chunks(int n) { return (n + 2 + ADJ_CHUNK - 1) / ADJ_CHUNK; }
__host__ __device__ inline int adj_groups(int nline, int nl) { return (nline + nl - 1) / nl; }
__host__ __device__ inline int adj_blocks(const Lay& L, int dir, int nl = ADJ_LINES) {
  return dir == 0 ? adj_groups(L.ny, nl) * adj_chunks(L.nx) : L.ny > 1 ? adj_groups(L.nx, nl) * adj_chunks(L.ny) : 0;
}
// Blocks of eight lines that three an SM hold at once.  Up to here the line kernels take 80 registers
// (three blocks an SM), above 64 with more spills (four).  A reverse step with four and with three, Euler /
// viscous with a body: 200x150 (302 blocks) 275 / 349 and 271 / 343 us, 250x190 (440) 339 / 418 and 333 /
// 410; 240x200 (465) 388 / 473 and 389 / 494, 256x200 (506) 398 / 480 and 402 / 502, 300x200 (579) 400 / 484
// and 414 / 506, 512x512 1332 / 1529 and 1340 / 1563; 16 instances 5.30 and 5.42 ms.  Two blocks (128
// registers, no spills): 512x512 viscous 1681.
constexpr int ADJ_THREE_BLOCKS = 3 * GB300_SMS;
// strips of a direction: [chunk][variable (5)][4 outer cells][line]
__host__ __device__ inline long long strip_size(const Lay& L, int dir) {
  return dir == 0 ? 20LL * adj_chunks(L.nx) * L.ny : L.ny > 1 ? 20LL * adj_chunks(L.ny) * L.nx : 0;
}
__device__ __forceinline__ double* strip(const AdjArgs& a, int dir, int chunk, int c, int e, int line) {
  const int nline = dir == 0 ? a.lay.ny : a.lay.nx;
  return a.strips + (dir == 0 ? 0 : strip_size(a.lay, 0)) + ((long long)(chunk * 5 + c) * 4 + e) * nline + line;
}

// block `item` of direction dir: ADJ_LINES warps, a line each (SPLIT: four warps a line, each with one
// variable's WENO5 forward and reverse, the first of them with the fluxes between); slot: the block's
// slot for its partials of pbar[0..3]; smem: adj_smem(SPLIT) doubles
template <bool VISC, bool SPLIT = false>
__device__ __forceinline__ void adj_lines(const AdjArgs& a, const double* __restrict__ Unext, double bdt, int dir,
                                          int item, double* smem, long long slot) {
  constexpr int NL = SPLIT ? ADJ_SPLIT : ADJ_LINES, AL = NL + 2, AP = adj_plane(NL);
  const Lay& L = a.lay;
  double* sq = smem;           // rho, u, v, p
  double* sl = smem + 4 * AP;  // Unext on fluid cells
  const Gas g = a.gas;
  const int nline = dir == 0 ? L.ny : L.nx, ncell = dir == 0 ? L.nx : L.ny;
  const int nch = adj_chunks(ncell);
  const int chunk = item % nch, line0 = item / nch * NL;
  const int i0 = -1 + ADJ_CHUNK * chunk;  // first reversed cell
  const int gyl = dir == 0 ? L.gy : 3, gyc = dir == 0 ? 3 : L.gy;  // ghost layers across / along the line
  for (int e = threadIdx.x; e < AP; e += 32 * ADJ_LINES) {
    // consecutive threads along x in both directions
    const int ln = dir == 0 ? e / AB : e % AL, pos = dir == 0 ? e % AB : e / AL;
    // past the array a line goes on with its outer cell's state (as in the stage kernel)
    const int line = line0 - 1 + ln, cell = imax(imin(i0 - 3 + pos, ncell + gyc - 1), -gyc);
    const bool in = line >= -gyl && line < nline + gyl;
    const int i = dir == 0 ? cell : line, j = dir == 0 ? line : cell;
    const long long t = in ? L.idx(i, j) : 0;
    double r = 1.0, u = 0.0, v = 0.0, p = 1.0, T;
    if (in) {
      r = a.X[t];
      cons_to_prim(r, a.X[L.plane + t], a.X[2 * L.plane + t], a.X[3 * L.plane + t], g, u, v, p, T);
    }
    const int o = ln * AB + pos;
    sq[o] = r;
    sq[AP + o] = u;
    sq[2 * AP + o] = v;
    sq[3 * AP + o] = p;
    const bool fluid = i >= 0 && i < L.nx && j >= 0 && j < L.ny && (a.tag == nullptr || a.tag[(long long)j * L.nx + i] == 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) sl[c * AP + o] = fluid ? Unext[c * L.plane + t] : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) / (SPLIT ? 4 : 1);
  const int kq = SPLIT ? (threadIdx.x >> 5) & 3 : 0;
  const int line = line0 + warp;
  const bool live = line < nline;
  double gs1 = 0.0, gs2 = 0.0, vmu = 0.0, vk = 0.0;
  if (SPLIT || live) {  // (the shared lines' warps meet at barriers)
    const ViscC& vc = dir == 0 ? a.vx : a.vy;
    const double fl = bdt * (dir == 0 ? a.inv_dx : a.inv_dy);  // lambda' differences over h
    const int pn = dir + 1, pt = 2 - dir;
    const bool inner = lane - 1u < 30u;
    const double* q = sq + (warp + 1) * AB + lane + 1;
    const double* l = sl + (warp + 1) * AB + lane + 1;
    const double* un = q + pn * AP;
    const double* ut = q + pt * AP;
    const int cell = i0 - 2 + lane, f = cell + 1;  // the lane's cell and its face at i+1/2
    const bool face = live && inner && lane < 30 && f >= 0 && f <= ncell;
    const bool own = lane >= 2;  // (with face) the warp's faces: lanes 2..29
    const bool rev = lane >= 2 && lane < 30;
    double* const ex = smem + 8 * AP + 12 * 32 * warp + lane;  // SPLIT: [12][32] of the line
    double bL[4], bR[4], dl[VISC ? 5 : 4], dr[VISC ? 5 : 4];
    bool fell = SPLIT;  // a face of the warp fell back to first order
    double Lq[4], Rq[4];
    if constexpr (SPLIT) {
      double Lf, Rf;
      weno_lane(q + ((kq == 1) ? pn : (kq == 2) ? pt : kq) * AP, 1, inner, Lf, Rf);
      ex[32 * kq] = Lf;
      ex[32 * (4 + kq)] = Rf;
      __syncthreads();
      if (kq == 0)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          Lq[m] = ex[32 * m];
          Rq[m] = ex[32 * (4 + m) + (lane < 31 ? 1 : 0)];
        }
    } else {
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        const int c = (k == 1) ? pn : (k == 2) ? pt : k;
        double Lf, Rf;
        weno_lane(q + c * AP, 1, inner, Lf, Rf);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          Lq[m] = (k == m) ? Lf : Lq[m];
          Rq[m] = (k == m) ? Rf : Rq[m];
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) Rq[m] = __shfl_down_sync(0xffffffffu, Rq[m], 1);
    }
    if (!SPLIT || kq == 0) {
      const bool fallback = !(positive(Lq[0]) && positive(Lq[3]) && positive(Rq[0]) && positive(Rq[3]));
      if (fallback) {
        Lq[0] = q[0], Lq[1] = un[0], Lq[2] = ut[0], Lq[3] = q[3 * AP];
        Rq[0] = q[1], Rq[1] = un[1], Rq[2] = ut[1], Rq[3] = q[3 * AP + 1];
      }
      double Fb[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const double* lm = l + (m == 1 ? pn : m == 2 ? pt : m) * AP;
        Fb[m] = (lm[1] - lm[0]) * fl;
      }
      double s1 = 0.0, s2 = 0.0;
      hllc_vjp(Lq, Rq, g, Fb, bL, bR, s1, s2);
      gs1 = own && face ? s1 : 0.0;
      gs2 = own && face ? s2 : 0.0;
      // adjoints that go straight to the cells of the warp's faces: left cell dl, right cell dr
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        dl[m] = fallback && face && own ? bL[m] : 0.0;
        dr[m] = fallback && face && own ? bR[m] : 0.0;
        bL[m] = fallback || !face ? 0.0 : bL[m];
        bR[m] = fallback || !face ? 0.0 : bR[m];
      }
      fell = __any_sync(0xffffffffu, fallback && face);
      if (VISC) {
        // F[n] -= tnn; F[t] -= tnt; F[3] -= 0.5 (sbn tnn + sbt tnt) + ck dT
        const double Tc = q[3 * AP] * recip(q[0]);
        const double dT = __shfl_down_sync(0xffffffffu, Tc, 1) - Tc;
        const double ua = un[0], ub = un[1], ta = ut[0], tb = ut[1];
        const double dun = ub - ua, dut = tb - ta;
        double tnn, tnt;
        if (a.two_d) {
          const double cun = un[AB] - un[-AB], cut = ut[AB] - ut[-AB];
          const double sun = cun + __shfl_down_sync(0xffffffffu, cun, 1), sut = cut + __shfl_down_sync(0xffffffffu, cut, 1);
          tnn = fma(vc.c43n, dun, -vc.c23t * sut);
          tnt = fma(vc.cn, dut, vc.ct * sun);
        } else {
          tnn = vc.c43n * dun;
          tnt = vc.cn * dut;
        }
        const double h3 = half_of(Fb[3]);
        const double btnn = fma(-h3, ua + ub, -Fb[1]), btnt = fma(-h3, ta + tb, -Fb[2]);
        const double bT = Fb[3] * vc.ck, ckk = -bT * dT;
        const double bdun = vc.c43n * btnn, bdut = vc.cn * btnt;
        if (own && face) {
          const double l1 = fma(-h3, tnn, -bdun), r1 = fma(-h3, tnn, bdun), l2 = fma(-h3, tnt, -bdut),
                       r2 = fma(-h3, tnt, bdut);
          if (fell) dl[1] += l1, dr[1] += r1, dl[2] += l2, dr[2] += r2;
          else dl[1] = l1, dr[1] = r1, dl[2] = l2, dr[2] = r2;
          vmu = fma(btnn, tnn, fma(btnt, tnt, ckk));
          vk = ckk;
        }
        dl[VISC ? 4 : 0] = own && face ? bT : 0.0;
        dr[VISC ? 4 : 0] = own && face ? -bT : 0.0;
        if (a.two_d) {
          // tangential differences: + to the cells one line up, minus to those one line down; the
          // cell's sum over its two faces
          const double xn = face ? vc.ct * btnt : 0.0, xt = face ? -vc.c23t * btnn : 0.0;
          const double tn = xn + __shfl_up_sync(0xffffffffu, xn, 1), tt = xt + __shfl_up_sync(0xffffffffu, xt, 1);
          if (live && rev && cell <= ncell) {
            double* o = a.tang + (long long)(2 * dir) * L.plane + (dir == 0 ? L.idx(cell, line) : L.idx(line, cell));
            o[0] = tn;
            o[L.plane] = tt;
          }
        }
      }
      if (a.fadj != nullptr && face) {
        const double* fa = a.fadj + (long long)(dir * 8) * a.splane + face_id(a, dir, f, line);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int c = (m == 1) ? pn : (m == 2) ? pt : m;
          bL[m] += fa[c * a.splane];
          bR[m] += fa[(4 + c) * a.splane];
        }
      }
      // the reversed cells' face states: L at i+1/2, R at i-1/2; right cells' straight terms
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const double up = __shfl_up_sync(0xffffffffu, bR[m], 1);
        bL[m] = rev ? bL[m] : 0.0;
        bR[m] = rev ? up : 0.0;
      }
      if (VISC || fell) {
#pragma unroll
        for (int m = 0; m < (VISC ? 5 : 4); ++m) {
          if ((m == 0 || m == 3) && !fell) continue;  // no such term
          const double up = __shfl_up_sync(0xffffffffu, dr[m], 1);
          dl[m] += lane > 0 ? up : 0.0;
        }
      }
    }
    if constexpr (SPLIT) {
      if (kq == 0) {
#pragma unroll
        for (int m = 0; m < 4; ++m) ex[32 * m] = bL[m], ex[32 * (4 + m)] = bR[m];
#pragma unroll
        for (int m = 0; m < 4; ++m) ex[32 * (8 + m)] = dl[m];
      }
      __syncthreads();
    }
    // where the lane's sums go: the cell's place, or a strip of the warp
    const bool in = live && cell >= -gyc && cell < ncell + gyc;
    double* qo = rev ? a.Qb + (long long)(dir * 5) * L.plane + (in ? (dir == 0 ? L.idx(cell, line) : L.idx(line, cell)) : 0)
                     : strip(a, dir, chunk, 0, lane < 2 ? lane : lane - 28, line);
    const long long qs = rev ? L.plane : 4LL * nline;
#pragma unroll 1
    for (int k = kq; k < (SPLIT ? kq + 1 : 4); ++k) {
      const int c = (k == 1) ? pn : (k == 2) ? pt : k;
      const double Lb = SPLIT ? ex[32 * k] : (k == 0) ? bL[0] : (k == 1) ? bL[1] : (k == 2) ? bL[2] : bL[3];
      const double Rb = SPLIT ? ex[32 * (4 + k)] : (k == 0) ? bR[0] : (k == 1) ? bR[1] : (k == 2) ? bR[2] : bR[3];
      double w[4];
      weno_grad_lane(q + c * AP, 1, inner, Lb, Rb, w);  // 0 where Lb = Rb = 0
      // adjoint of d_{i+1/2}: its share in the reversed cells i-1 .. i+2
      const double u3 = __shfl_up_sync(0xffffffffu, w[3], 1);
      const double t = (w[2] + (lane > 0 ? u3 : 0.0)) +
                       (__shfl_down_sync(0xffffffffu, w[1], 1) + __shfl_down_sync(0xffffffffu, w[0], 2));
      const double tm = __shfl_up_sync(0xffffffffu, t, 1);
      double v = fma(SIXTH, (lane > 0 ? tm : 0.0) - t, Lb + Rb);
      if (fell || (VISC && (k == 1 || k == 2))) v += SPLIT ? ex[32 * (8 + k)] : (k == 0) ? dl[0] : (k == 1) ? dl[1] : (k == 2) ? dl[2] : dl[3];
      if (in) qo[c * qs] = v;
    }
    if (VISC && in && (!SPLIT || kq == 0)) qo[4 * qs] = dl[VISC ? 4 : 0];
  }
  if (a.pp == nullptr) return;
  // gamma, mu and Pr from the block's sums
  const double t = block_sum4(gs1, gs2, vmu, vk);
  if (threadIdx.x < 4) {
    const double s1 = __shfl_sync(0xfu, t, 0), s2 = __shfl_sync(0xfu, t, 1), sm = __shfl_sync(0xfu, t, 2), sk = __shfl_sync(0xfu, t, 3);
    const double gb = s2 / g.gamma - s1 * g.g1 * g.g1;
    a.pp[4 * slot + threadIdx.x] =
        threadIdx.x == 0 ? (VISC ? fma(a.kg, sk, gb) : gb) : !VISC || threadIdx.x == 3 ? 0.0 : threadIdx.x == 1 ? sm * a.inv_mu : sk * a.kp;
  }
}

// the line sums of primitive c at padded cell (i, j)
template <int DIR>
__device__ __forceinline__ double line_sum(const AdjArgs& a, int c, int i, int j) {
  const Lay& L = a.lay;
  const int m = DIR == 0 ? i : j, line = DIR == 0 ? j : i;
  const int n = DIR == 0 ? L.nx : L.ny, nch = adj_chunks(n);
  if (m < -1) return *strip(a, DIR, 0, c, m + 3, line);  // cells -3, -2: the first warp's strip
  const int ch = (m + 1) / ADJ_CHUNK, pos = (m + 1) % ADJ_CHUNK;
  double v = ch < nch ? a.Qb[(long long)(DIR * 5 + c) * L.plane + L.idx(i, j)] : 0.0;
  if (pos < 2 && ch > 0) v += *strip(a, DIR, ch - 1, c, 2 + pos, line);
  if (pos >= ADJ_CHUNK - 2 && ch + 1 < nch) v += *strip(a, DIR, ch + 1, c, pos - (ADJ_CHUNK - 2), line);
  return v;
}

// Ub of padded cell t (all four planes); gamma and nu contributions are added to gb, nb
template <bool VISC>
__device__ __forceinline__ void adj_cell(const AdjArgs& a, const double* __restrict__ Unext, double* __restrict__ Uacc,
                                         double ra, double rb, double bdt, int rhs_mode, long long t, double& gb,
                                         double& nb) {
  const Lay& L = a.lay;
  if (t >= L.plane) return;
  const int col = (int)(t % L.pitch), row = (int)(t / L.pitch);
  if (col >= L.nx + 6 || row >= L.H) return;
  const int i = col - 3, j = row - L.gy;
  const bool xl = j >= 0 && j < L.ny, yl = a.two_d && i >= 0 && i < L.nx;  // on an x / a y line
  double qb[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, ub[4];
#pragma unroll
  for (int c = 0; c < (VISC ? 5 : 4); ++c) {
    if (xl) qb[c] += line_sum<0>(a, c, i, j);
    if (yl) qb[c] += line_sum<1>(a, c, i, j);
  }
  if (VISC && a.two_d) {
    // tangential terms: from the line below and, negative, from the line above (cells -1 .. n of them)
    const double* tx = a.tang;
    const double* ty = a.tang + 2 * L.plane;
    if (i >= -1 && i <= L.nx) {
      if (j - 1 >= 0 && j - 1 < L.ny) qb[1] += tx[t - L.pitch], qb[2] += tx[L.plane + t - L.pitch];
      if (j + 1 >= 0 && j + 1 < L.ny) qb[1] -= tx[t + L.pitch], qb[2] -= tx[L.plane + t + L.pitch];
    }
    if (j >= -1 && j <= L.ny) {
      if (i - 1 >= 0 && i - 1 < L.nx) qb[2] += ty[t - 1], qb[1] += ty[L.plane + t - 1];
      if (i + 1 >= 0 && i + 1 < L.nx) qb[2] -= ty[t + 1], qb[1] -= ty[L.plane + t + 1];
    }
  }
  double u, v, p, T;
  const double r = a.X[t];
  cons_to_prim(r, a.X[L.plane + t], a.X[2 * L.plane + t], a.X[3 * L.plane + t], a.gas, u, v, p, T);
  prim_vjp(r, u, v, p, a.gas, qb, ub, gb);
  auto fluid_at = [&](int x, int y) {
    return x >= 0 && x < L.nx && y >= 0 && y < L.ny && (a.tag == nullptr || a.tag[(long long)y * L.nx + x] == 0);
  };
  const bool interior = i >= 0 && i < L.nx && j >= 0 && j < L.ny, fluid = fluid_at(i, j);
  if (a.has_av && i >= -1 && i <= L.nx && j >= (a.two_d ? -1 : 0) && j <= (a.two_d ? L.ny : 0)) {
    const bool xm = fluid_at(i - 1, j), xp = fluid_at(i + 1, j), ym = a.two_d && fluid_at(i, j - 1),
               yp = a.two_d && fluid_at(i, j + 1);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double* lp = Unext + c * L.plane + t;
      const double l0 = fluid ? lp[0] : 0.0;
      double add = a.nu_x * (((xm ? lp[-1] : 0.0) - 2.0 * l0) + (xp ? lp[1] : 0.0));
      if (a.two_d) add += a.nu_y * (((ym ? lp[-L.pitch] : 0.0) - 2.0 * l0) + (yp ? lp[L.pitch] : 0.0));
      ub[c] = fma(bdt, add, ub[c]);
      if (fluid && l0 != 0.0) {
        const double* X = a.X + c * L.plane;
        double lap = a.nu_x1 * ((X[t - 1] - 2.0 * X[t]) + X[t + 1]);
        if (a.two_d) lap += a.nu_y1 * ((X[t - L.pitch] - 2.0 * X[t]) + X[t + L.pitch]);
        nb += bdt * l0 * lap;
      }
    }
  }
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

// =======================================================================================
// transposed halo fill (gathers).  y sides first: targets are cells of interior rows (all
// padded columns); then x sides: targets are interior cells.
// =======================================================================================
__device__ __forceinline__ void adj_bcT_one(const AdjArgs& a, const BcArgs& bc, int phase_y, double* inflow_part,
                                            int tmax, long long t) {
  const Lay& L = a.lay;
  // targets: 6 source rows/columns next to each boundary, a run of ntan threads each (a warp takes
  // one branch; along a row its loads are consecutive)
  const int ntan = phase_y ? L.nx + 6 : L.ny;
  const int r = (int)(t / ntan);
  const int tpos = (int)(t - (long long)r * ntan), tan = tpos - (phase_y ? 3 : 0);
  const int n = phase_y ? L.ny : L.nx;
  if (r < 6) {
    const int tgt = (r < 3) ? r : n - 6 + r;  // 0,1,2, n-3,n-2,n-1
    const int comp = phase_y ? 2 : 1;          // momentum component normal to the side
    const long long tid = phase_y ? L.idx(tan, tgt) : L.idx(tgt, tan);
    double acc[4] = {0.0, 0.0, 0.0, 0.0}, own[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) own[c] = a.Ub[c * L.plane + tid];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int kind = bc.kind[(phase_y ? 2 : 0) + s];
      // the halo layers k = ka .. kb of this side that copy the target row
      int ka, kb;
      if (kind == 0) {
        ka = 1;
        kb = (tgt == (s == 0 ? 0 : n - 1)) ? 3 : 0;
      } else {
        const bool near_low = (kind == 1) == (s == 0);  // layer k holds row k - 1, else n - k
        ka = kb = near_low ? tgt + 1 : n - tgt;
      }
      if (kind == 3 || ka > 3 || kb < ka) continue;
      double h[3][4];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int l = min(ka + k, kb), hl = (s == 0) ? -l : n - 1 + l;
        const long long hid = phase_y ? L.idx(tan, hl) : L.idx(hl, tan);
#pragma unroll
        for (int c = 0; c < 4; ++c) h[k][c] = a.Ub[c * L.plane + hid];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (ka + k <= kb)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[c] += (kind == 1 && c == comp) ? -h[k][c] : h[k][c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) a.Ub[c * L.plane + tid] = own[c] + acc[c];
  } else if (r < 8) {
    // inflow sides: the halo adjoints of each (side, tangential position), its three layers in
    // order, into inflow_part[side][position] (summed over positions by adj_inflow_block)
    const int s = r - 6, side = (phase_y ? 2 : 0) + s;
    if (bc.kind[side] != 3) return;
    double h[3][4];
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
      const int hl = (s == 0) ? -k : n - 1 + k;
      const long long hid = phase_y ? L.idx(tan, hl) : L.idx(hl, tan);
#pragma unroll
      for (int c = 0; c < 4; ++c) h[k - 1][c] = a.Ub[c * L.plane + hid];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      inflow_part[((long long)side * tmax + tpos) * 4 + c] = ((0.0 + h[0][c]) + h[1][c]) + h[2][c];
  }
}

// inflow halo adjoints (conserved) -> gradient of the inflow primitive state and gamma; one
// warp per side sums its partials in a fixed order, then one thread adds to pbar side by side
// S[side] = the sums of a side's inflow halo adjoints (warp `side` of the first four)
__device__ __forceinline__ void adj_inflow_sums(const AdjArgs& a, const BcArgs& bc, const double* inflow_part, int tmax,
                                                double S[4][4]) {
  const int side = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Lay& L = a.lay;
  if (side < 4 && bc.kind[side] == 3) {
    const int ntan = (side < 2) ? L.ny : L.nx + 6;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int k = lane; k < ntan; k += 32)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] += inflow_part[((long long)side * tmax + k) * 4 + c];
    const double t = warp_sum4(v[0], v[1], v[2], v[3]);
    if ((lane & 7) == 0) S[side][lane >> 3] = t;
  }
}
// the inflow states' gradient, a thread (of the first 16) per side and parameter, from
// U = (r, r u, r v, p/(gamma-1) + r (u^2 + v^2)/2)
__device__ __forceinline__ void adj_inflow_states(const AdjArgs& a, const BcArgs& bc, const double* inflow_prim,
                                                  const double S[4][4]) {
  if (threadIdx.x >= 16 || bc.kind[threadIdx.x >> 2] != 3) return;
  const int sd = threadIdx.x >> 2, m = threadIdx.x & 3;
  const double* s = S[sd];
  const double r = inflow_prim[4 * sd], u = inflow_prim[4 * sd + 1], v = inflow_prim[4 * sd + 2];
  a.pbar[4 + 4 * sd + m] += pick4(m, s[0] + s[1] * u + s[2] * v + s[3] * 0.5 * (u * u + v * v), s[1] * r + s[3] * r * u,
                                  s[2] * r + s[3] * r * v, s[3] * a.gas.g1);
}
// and their part of gamma's
__device__ __forceinline__ double adj_inflow_gamma(const AdjArgs& a, const BcArgs& bc, const double* inflow_prim,
                                                   const double S[4][4]) {
  double g = 0.0;
  for (int sd = 0; sd < 4; ++sd)
    if (bc.kind[sd] == 3) g += -S[sd][3] * inflow_prim[4 * sd + 3] * a.gas.g1 * a.gas.g1;
  return g;
}
__device__ __forceinline__ void adj_inflow_block(const AdjArgs& a, const BcArgs& bc, const double* inflow_part,
                                                 int tmax, const double* inflow_prim) {
  __shared__ double S[4][4];
  if (a.pbar != nullptr) adj_inflow_sums(a, bc, inflow_part, tmax, S);
  __syncthreads();
  if (a.pbar == nullptr) return;
  adj_inflow_states(a, bc, inflow_prim, S);
  if (threadIdx.x == 32) a.pbar[0] += adj_inflow_gamma(a, bc, inflow_prim, S);
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
#pragma unroll 4
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
// item t = 4 k + m: ghost k, lane m of a quad
__device__ __forceinline__ void adj_ib_ghost_one(const AdjArgs& a, const IbArgs& ib, int wall, double* qIb, int t,
                                                 double& gb) {
  if (t < 4 * ib.n) {
    const int k = t >> 2, m = t & 3;
    const Lay& L = a.lay;
    const long long d = m * L.plane + ib.dst[k];
    const double own = a.Ub[d];
    a.Ub[d] = 0.0;  // the ghost's own input value is overwritten by the fill
    double q[4], nx, ny, ug, vg;
    ib_image(a.X, L, ib, a.gas.gm1, wall, k, m, q, nx, ny, ug, vg);
    double G[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) G[c] = __shfl_sync(0xfu << (threadIdx.x & 28), own, c, 4);
    // G = (r, r ug, r vg, p/(gamma-1) + r (ug^2 + vg^2)/2)
    const double br = G[0] + G[1] * ug + G[2] * vg + G[3] * 0.5 * (ug * ug + vg * vg);
    const double bug = G[1] * q[0] + G[3] * q[0] * ug;
    const double bvg = G[2] * q[0] + G[3] * q[0] * vg;
    const double g1 = a.gas.g1;
    if (m == 0) gb -= G[3] * q[3] * g1 * g1;
    double bu, bv;
    if (wall == 0) {  // (ug, vg) = (I - 2 n n^T)(u, v): symmetric
      const double bn = bug * nx + bvg * ny;
      bu = bug - 2.0 * bn * nx;
      bv = bvg - 2.0 * bn * ny;
    } else {
      bu = -bug;
      bv = -bvg;
    }
    qIb[t] = pick4(m, br, bu, bv, G[3] * g1);
  }
}

// item t = 4 s + m: source cell s, lane m of a quad sums and writes component m
__device__ __forceinline__ void adj_ib_src_one(const AdjArgs& a, const IbTArgs& tb, const double* qIb, int t,
                                               double& gb) {
  if (t < 4 * tb.nsrc) {
    const int s = t >> 2, m = t & 3;
    const Lay& L = a.lay;
    const long long id = tb.cell[s];
    const int e0 = tb.ptr[s], e1 = tb.ptr[s + 1];
    const double r = a.X[id], mx = a.X[L.plane + id], my = a.X[2 * L.plane + id], E = a.X[3 * L.plane + id];
    const double own = a.Ub[m * L.plane + id];
    double sm = 0.0;
#pragma unroll 4
    for (int e = e0; e < e1; ++e) sm += tb.w[e] * qIb[4 * tb.ghost[e] + m];
    double S[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 4; ++c) S[c] = __shfl_sync(0xfu << (threadIdx.x & 28), sm, c, 4);
    double ub[4], u, v, p, T, g = 0.0;
    cons_to_prim(r, mx, my, E, a.gas, u, v, p, T);
    prim_vjp(r, u, v, p, a.gas, S, ub, g);
    if (m == 0) gb += g;
    a.Ub[m * L.plane + id] = own + pick4(m, ub[0], ub[1], ub[2], ub[3]);
  }
}

// =======================================================================================
// small elementwise helpers
// =======================================================================================
// cell t (fewer than 2^31), its four planes
__device__ __forceinline__ void adj_unpack_add_one(const double* __restrict__ P, const double* __restrict__ P2,
                                                   double* __restrict__ U, const Lay& lay, unsigned t) {
  const unsigned n = (unsigned)lay.nx * (unsigned)lay.ny;
  if (t >= n) return;
  const int i = (int)(t % (unsigned)lay.nx), j = (int)(t / (unsigned)lay.nx);
  const long long id = lay.idx(i, j);
  double v[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = P2 ? P[c * lay.plane + id] + P2[c * lay.plane + id] : P[c * lay.plane + id];
#pragma unroll
  for (int c = 0; c < 4; ++c) U[(long long)c * n + t] = v[c];
}

}  // namespace js
