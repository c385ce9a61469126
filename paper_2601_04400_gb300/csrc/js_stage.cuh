// One stage of the FP64 finite-volume step (arXiv 2601.04400, Sec. 2) in two launches: lines (the
// flux differences of every x and y line: primitives, WENO5, HLLC, viscous flux) and cells (their
// divergence, artificial viscosity and the SSP-RK3 stage combination).  Used by the per-grid kernels
// and by the batched ones.
//
// A warp takes 28 cells of one line, a lane one cell: what a cell shares with its neighbours
// (differences, smoothness indicators, face states, face fluxes) is passed by shuffles.  Of the 32
// cells of lanes 0..31 (cells -2 .. 29 of the 28) the differences serve WENO5 of cells -1 .. 28, these
// the faces -1/2 .. 27 1/2, these the 28 outputs.  No state is carried along a line, so a thread holds
// one cell's values (64 registers; sweeping 16 cells with a sliding window in registers took 214 and
// left 2 warps per SM sub-partition, too few to overlap the integer WENO5 with the FP64 of the
// fluxes), and a line takes one pass of latency instead of 17.
//
// Lines are independent of one another: no barrier but the one after the block's loads, and work in
// units of 8 lines.  (Fused 28x28 tiles, x and y lines of a tile and its combination in one block with
// the flux differences in shared memory, lost 18% of their warps' time to barriers and up to a quarter
// to the last wave: 1369 tiles of a 1024^2 grid on 456 resident blocks take four waves.)  The flux
// differences cost 128 bytes a cell of memory traffic, mostly in the L2.
#pragma once
#include <type_traits>

#include "js_device.cuh"
#include "js_internal.h"

namespace js {

constexpr unsigned FULL = 0xffffffffu;
__device__ __forceinline__ u64 shfl_up(u64 v) { return (u64)__shfl_up_sync(FULL, (unsigned long long)v, 1); }
__device__ __forceinline__ u64 shfl_down(u64 v) { return (u64)__shfl_down_sync(FULL, (unsigned long long)v, 1); }
__device__ __forceinline__ double shfl_up(double v) { return __shfl_up_sync(FULL, v, 1); }
__device__ __forceinline__ double shfl_down(double v) { return __shfl_down_sync(FULL, v, 1); }

struct NoFace {
  __device__ __forceinline__ void operator()(const double*, const double*) const {}
};

// Flux differences F_{i+1/2} - F_{i-1/2} (conserved order) of the cell q points at (planes rho, u,
// v, p, and T when VISC, `ps` apart; neighbours along the line at q[-1], q[1], across it at q[-ts],
// q[ts]), valid in lanes 2..29.  pn: plane of the face-normal velocity (1 or 2).  Every lane of the
// warp calls it, consecutive lanes on consecutive cells; q[-1 .. 1] is readable for each.
// face(ql, qr), when given, receives the two WENO5 states of face i+1/2 before any positivity
// fallback (lanes 1..29).
// fb null: the warp takes the line alone.  Else four warps share it, warp k (of the block's, mod 4)
// reconstructing variable k into fb ([8][32], one per line) and warp 0 going on after a barrier of the
// block: the same values with a quarter of the reconstructions' latency.  False for the other warps.
template <bool VISC, bool HAS_T, class Face = NoFace>
__device__ __forceinline__ bool line_fluxes(const double* q, int ps, int ts, int pn, const Gas& g, const ViscC& vc,
                                            double dF[4], double* fb, Face face = Face{}) {
  constexpr bool FI = !std::is_same<Face, NoFace>::value;
  constexpr int st = 1;
  const int lane = threadIdx.x & 31;
  const bool inner = lane - 1u < 30u;
  const int pt = 3 - pn;
  // face states of the cell in the line's frame: rho, normal, tangential velocity, p
  double L[4], R[4];
  if (fb != nullptr) {
    const int k = (threadIdx.x >> 5) & 3;
    double Lf, Rf;
    weno_lane(q + ((k == 1) ? pn : (k == 2) ? pt : k) * ps, st, inner, Lf, Rf);
    fb[32 * k + lane] = Lf;
    fb[32 * (4 + k) + lane] = Rf;
    __syncthreads();
    if (k != 0) return false;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      L[m] = fb[32 * m + lane];
      R[m] = fb[32 * (4 + m) + min(lane + 1, 31)];
    }
  } else {
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
      const int c = (k == 1) ? pn : (k == 2) ? pt : k;
      double Lf, Rf;
      weno_lane(q + c * ps, st, inner, Lf, Rf);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        L[m] = (k == m) ? Lf : L[m];
        R[m] = (k == m) ? Rf : R[m];
      }
    }
    // face i+1/2: the cell's left-biased state, its neighbour's right-biased one
#pragma unroll
    for (int m = 0; m < 4; ++m) R[m] = shfl_down(R[m]);
  }
  const double* un = q + pn * ps;
  const double* ut = q + pt * ps;
  if (FI) {
    const double ql[4] = {L[0], pn == 1 ? L[1] : L[2], pn == 1 ? L[2] : L[1], L[3]};
    const double qr[4] = {R[0], pn == 1 ? R[1] : R[2], pn == 1 ? R[2] : R[1], R[3]};
    face(ql, qr);
  }
  if (!(positive(L[0]) && positive(L[3]) && positive(R[0]) && positive(R[3]))) {
    // positivity fallback: first-order (cell) states at this face
    L[0] = q[0], L[1] = un[0], L[2] = ut[0], L[3] = q[3 * ps];
    R[0] = q[st], R[1] = un[st], R[2] = ut[st], R[3] = q[3 * ps + st];
  }
  double F[4];
  hllc(L[0], L[1], L[2], L[3], R[0], R[1], R[2], R[3], g, F);
  if (VISC) {
    const double* Tq = q + 4 * ps;
    const double ua = un[0], ub = un[st], ta = ut[0], tb = ut[st];
    const double dun = ub - ua, dut = tb - ta, dT = Tq[st] - Tq[0];
    double tnn, tnt;
    if (HAS_T) {
      const double cun = un[ts] - un[-ts], cut = ut[ts] - ut[-ts];
      const double sun = cun + shfl_down(cun), sut = cut + shfl_down(cut);
      tnn = fma(vc.c43n, dun, -vc.c23t * sut);
      tnt = fma(vc.cn, dut, vc.ct * sun);
    } else {
      tnn = vc.c43n * dun;
      tnt = vc.cn * dut;
    }
    const double sbn = ua + ub, sbt = ta + tb;
    F[1] -= tnn;
    F[2] -= tnt;
    F[3] = fma(-0.5, fma(sbn, tnn, sbt * tnt), fma(-vc.ck, dT, F[3]));
  }
  double D[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) D[m] = F[m] - shfl_up(F[m]);
  dF[0] = D[0];
  dF[1] = pn == 1 ? D[1] : D[2];
  dF[2] = pn == 1 ? D[2] : D[1];
  dF[3] = D[3];
  return true;
}

// =======================================================================================
// lines
// =======================================================================================
constexpr int SCHUNK = 28, SLINES = 8;  // cells a warp, lines (warps) a block
constexpr int SB = SCHUNK + 6;          // positions of a line's box: lane l at l + 1
constexpr int SPLIT_LINES = SLINES / 4;  // lines a block where four warps share one
// plane of a block's box, [line][position] in both directions: nl lines and one on either side
__host__ __device__ constexpr int stage_plane(int nl) { return SB * (nl + 2); }

__host__ __device__ inline int stage_chunks(int n) { return (n + SCHUNK - 1) / SCHUNK; }
__host__ __device__ inline int stage_blocks(const Lay& L, int dir, int nl = SLINES) {
  return dir == 0 ? (L.ny + nl - 1) / nl * stage_chunks(L.nx) : (L.nx + nl - 1) / nl * stage_chunks(L.ny);
}
template <bool VISC, bool SPLIT = false>
__host__ __device__ constexpr size_t stage_smem() {
  return sizeof(double) * (size_t)((VISC ? 5 : 4) * stage_plane(SPLIT ? SPLIT_LINES : SLINES) + (SPLIT ? SPLIT_LINES * 256 : 0));
}

// face image of the neural flux (IMG: a.img, FP32 [4][ny][nx+1] for x faces then [4][nx][ny+1]
// for y faces): face f of a line
__device__ __forceinline__ void put_image(const StageArgs& a, int dir, int line, int f, const double* ql,
                                          const double* qr) {
  const int nx = a.lay.nx, ny = a.lay.ny;
  const long long pix0 = (long long)ny * (nx + 1);
  const long long pix = (dir == 0) ? pix0 : (long long)nx * (ny + 1);
  float* X = a.img + (dir == 0 ? 0LL : 4 * pix0) + (long long)line * ((dir == 0 ? nx : ny) + 1) + f;
  const double wl[4] = {ql[0], dir == 0 ? ql[1] : ql[2], dir == 0 ? ql[2] : ql[1], ql[3]};
  const double wr[4] = {qr[0], dir == 0 ? qr[1] : qr[2], dir == 0 ? qr[2] : qr[1], qr[3]};
  float m[4];
  face_image<float>(wl, wr, 1, 2, a.img_g1, a.img_mean, a.img_isd, m);
#pragma unroll
  for (int k = 0; k < 4; ++k) X[k * pix] = m[k];
}

// block `item` of direction dir (0: x lines): SLINES warps, a line each (SPLIT: four warps a line);
// writes the flux differences to a.dF (4 padded planes for x, 4 for y)
template <bool VISC, bool IMG, bool SPLIT = false>
__device__ __forceinline__ void stage_lines(const StageArgs& a, int dir, int item, double* sq) {
  constexpr int NL = SPLIT ? SPLIT_LINES : SLINES, SL = NL + 2, SP = stage_plane(NL);
  const Lay& L = a.lay;
  const Gas g{a.gamma, a.gm1, a.g1};
  const int nline = dir == 0 ? L.ny : L.nx, ncell = dir == 0 ? L.nx : L.ny;
  const int nch = stage_chunks(ncell);
  const int i0 = SCHUNK * (item % nch), line0 = item / nch * NL;
  const int gyl = dir == 0 ? L.gy : 3, gyc = dir == 0 ? 3 : L.gy;  // ghost layers across / along the line
  for (int e = threadIdx.x; e < SP; e += 32 * SLINES) {
    // consecutive threads along x in both directions
    const int ln = dir == 0 ? e / SB : e % SL, pos = dir == 0 ? e % SB : e / SL;
    if (!VISC && (ln == 0 || ln == SL - 1)) continue;  // lines beside the block's own serve the viscous terms
    const int line = line0 - 1 + ln, cell = imin(i0 - 3 + pos, ncell + gyc - 1);
    // past the array a line goes on with its last cell's state and the lines beyond hold a uniform one (they
    // feed only cells that are not written; a jump there would part the warp in weno_faces)
    const bool in = line >= -gyl && line < nline + gyl;
    double r = 1.0, u = 0.0, v = 0.0, p = 1.0, T = 1.0;
    if (in) {
      const long long t = dir == 0 ? L.idx(cell, line) : L.idx(line, cell);
      r = a.Uin[t];
      cons_to_prim(r, a.Uin[L.plane + t], a.Uin[2 * L.plane + t], a.Uin[3 * L.plane + t], g, u, v, p, T);
    }
    const int o = ln * SB + pos;
    sq[o] = r;
    sq[SP + o] = u;
    sq[2 * SP + o] = v;
    sq[3 * SP + o] = p;
    if (VISC) sq[4 * SP + o] = T;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, ln = (threadIdx.x >> 5) / (SPLIT ? 4 : 1);
  const int line = line0 + ln, cell = i0 - 2 + lane;
  if (!SPLIT && line >= nline) return;  // (the shared lines' warps meet at a barrier)
  const double* q = sq + (ln + 1) * SB + lane + 1;
  double* const fb = SPLIT ? sq + (VISC ? 5 : 4) * SP + 256 * ln : nullptr;
  double dF[4];
  const ViscC& vc = dir == 0 ? a.vx : a.vy;
  if constexpr (IMG) {
    const bool mine = line_fluxes<VISC, true>(q, SP, SB, dir + 1, g, vc, dF, fb, [&](const double* ql, const double* qr) {
      // face cell + 1; the chunk's outer face belongs to the next chunk unless it is the line's last
      const int f = cell + 1;
      if (line < nline && lane >= 1 && f <= ncell && (lane <= 28 || (lane == 29 && f == ncell))) put_image(a, dir, line, f, ql, qr);
    });
    if (!mine) return;
  } else {
    if (!line_fluxes<VISC, true>(q, SP, SB, dir + 1, g, vc, dF, fb)) return;
  }
  if (line < nline && lane >= 2 && lane < 30 && cell < ncell) {
    const int i = dir == 0 ? cell : line, j = dir == 0 ? line : cell;
    const long long t = L.idx(i, j);
    if (dir == 0 && !(positive(q[0]) && positive(q[3 * SP])) &&
        (a.tag == nullptr || a.tag[(long long)j * L.nx + i] == 0))
      atomicOr(a.err, ERR_NONPHYSICAL_BIT);
    double* D = a.dF + (long long)(4 * dir) * L.plane + t;
#pragma unroll
    for (int c = 0; c < 4; ++c) D[c * L.plane] = dF[c];
  }
}

// =======================================================================================
// cells
// =======================================================================================
// interior cell (gi, gj) from its flux differences dF, dG (dG unused in 1D)
template <bool RHS>
__device__ __forceinline__ void finish_cell(const StageArgs& a, int gi, int gj, const double dF[4], const double dG[4]) {
  const long long pid = a.lay.idx(gi, gj);
  const bool fluid = (a.tag == nullptr) || (a.tag[(long long)gj * a.lay.nx + gi] == 0);
  double out[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const double* Uc = a.Uin + c * a.lay.plane;
    const double us = RHS && fluid ? 0.0 : Uc[pid];
    double v = fma(-a.cx, dF[c], us);
    if (a.lay.ny > 1) v = fma(-a.cy, dG[c], v);
    if (a.has_av) {
      v = fma(a.avx, (Uc[pid + 1] - 2.0 * Uc[pid]) + Uc[pid - 1], v);
      if (a.lay.ny > 1) v = fma(a.avy, (Uc[pid + a.lay.pitch] - 2.0 * Uc[pid]) + Uc[pid - a.lay.pitch], v);
    }
    if (!RHS && a.use_un) v = fma(a.rk_a, a.Un[c * a.lay.plane + pid], a.rk_b * v);
    out[c] = fluid ? v : RHS ? 0.0 : us;
  }
  if (RHS) {
    const long long n = (long long)a.lay.nx * a.lay.ny;
    const long long o = (long long)gj * a.lay.nx + gi;
#pragma unroll
    for (int c = 0; c < 4; ++c) a.Uout[c * n + o] = out[c];
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) a.Uout[c * a.lay.plane + pid] = out[c];
  }
}

template <bool RHS>
__device__ __forceinline__ void stage_cell(const StageArgs& a, int gi, int gj) {
  const double* D = a.dF + a.lay.idx(gi, gj);
  double dF[4], dG[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    dF[c] = D[c * a.lay.plane];
    dG[c] = D[(4 + c) * a.lay.plane];
  }
  finish_cell<RHS>(a, gi, gj, dF, dG);
}

}  // namespace js
