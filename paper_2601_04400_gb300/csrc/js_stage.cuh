// Fused stage of the FP64 finite-volume step on one 2D tile (arXiv 2601.04400, Sec. 2):
// conserved tile + 3-cell halo -> primitives in shared memory -> fluxes of the tile's x lines,
// then of its y lines (WENO5, HLLC, viscous flux) -> divergence, artificial viscosity and the
// SSP-RK3 stage combination.  Used by the per-grid stage kernels and by the persistent batched
// kernels.
//
// A warp takes one line of the tile, a lane one cell of it: what a cell shares with its
// neighbours (differences, smoothness indicators, face states, face fluxes) is passed by
// shuffles.  Of the 32 cells of lanes 0..31 (cells -2 .. 29 of the line's 28 output cells) the
// differences serve WENO5 of cells -1 .. 28, these the faces -1/2 .. 27 1/2, these the 28 outputs.
// No state is carried along a line, so a thread holds one cell's values (about 100 registers;
// sweeping 16 cells with a sliding window in registers took 214 and left 2 warps per SM
// sub-partition, too few to overlap the integer WENO5 with the FP64 of the fluxes), and a line
// takes one pass of latency instead of 17.  28 of 32 lanes' work is kept.
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
// v, p, and T when VISC, `ps` apart; neighbours along the line at multiples of st, across it of
// ts), valid in lanes 2..29.  pn: plane of the face-normal velocity (1 or 2).  Every lane of the
// warp calls it, consecutive lanes on consecutive cells; q[-st .. st] is readable for each.
// face(ql, qr), when given, receives the two WENO5 states of face i+1/2 before any positivity
// fallback (lanes 1..29).
template <bool VISC, bool HAS_T, class Face = NoFace>
__device__ __forceinline__ void line_fluxes(const double* q, int ps, int st, int ts, int pn, const Gas& g,
                                            const ViscC& vc, double dF[4], Face face = Face{}) {
  constexpr bool FI = !std::is_same<Face, NoFace>::value;
  const int lane = threadIdx.x & 31;
  const bool inner = lane - 1u < 30u;
  const int pt = 3 - pn;
  // face states of the cell in the line's frame: rho, normal, tangential velocity, p
  double L[4], R[4];
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    const int c = (k == 1) ? pn : (k == 2) ? pt : k;
    double Lf, Rf;
    weno_lane(q + c * ps, st, k == 0 || k == 3, inner, Lf, Rf);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      L[m] = (k == m) ? Lf : L[m];
      R[m] = (k == m) ? Rf : R[m];
    }
  }
  // face i+1/2: the cell's left-biased state, its neighbour's right-biased one
#pragma unroll
  for (int m = 0; m < 4; ++m) R[m] = shfl_down(R[m]);
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
      const double sun = (un[ts] - un[-ts]) + (un[st + ts] - un[st - ts]);
      const double sut = (ut[ts] - ut[-ts]) + (ut[st + ts] - ut[st - ts]);
      tnn = fma(vc.c43n, dun, -vc.c23t * sut);
      tnt = fma(vc.cn, dut, vc.ct * sun);
    } else {
      tnn = vc.c43n * dun;
      tnt = vc.cn * dut;
    }
    const double sbn = ua + ub, sbt = ta + tb;
    const double e = fma(0.5, fma(sbn, tnn, sbt * tnt), vc.ck * dT);
    F[1] -= tnn;
    F[2] -= tnt;
    F[3] -= e;
  }
  double D[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) D[m] = F[m] - shfl_up(F[m]);
  dF[0] = D[0];
  dF[1] = pn == 1 ? D[1] : D[2];
  dF[2] = pn == 1 ? D[2] : D[1];
  dF[3] = D[3];
}

// =======================================================================================
// tiles
// =======================================================================================
constexpr int TILE = 28;         // output cells of a tile along x and along y (one warp's lines)
constexpr int TILE_B = TILE + 6;  // its box with the halo; the TMA copy writes dense rows
constexpr int TILE_A = TILE + 1;  // row pitch of the accumulator (odd: y lines hit distinct banks)

template <bool VISC>
struct StageTile {
  static constexpr int NPL = VISC ? 5 : 4;
  static constexpr int PS = TILE_B * TILE_B;
  static constexpr int PA = TILE * TILE_A;
  static constexpr size_t SMEM = sizeof(double) * (size_t)(NPL * PS + 4 * PA);
};

// final combination for one interior cell, v = U_s - dt div F (RHS mode: - div F)
template <bool RHS>
__device__ __forceinline__ void finish_cell(const StageArgs& a, int gi, int gj, const double upd[4], double rho,
                                            double p) {
  const long long pid = a.lay.idx(gi, gj);
  const bool fluid = (a.tag == nullptr) || (a.tag[(long long)gj * a.lay.nx + gi] == 0);
  double out[4];
  if (fluid) {
    if (!(positive(rho) && positive(p))) atomicOr(a.err, ERR_NONPHYSICAL_BIT);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double* Uc = a.Uin + c * a.lay.plane;
      double v = upd[c];
      if (a.has_av) {
        v = fma(a.avx, (Uc[pid + 1] - 2.0 * Uc[pid]) + Uc[pid - 1], v);
        if (a.lay.ny > 1) v = fma(a.avy, (Uc[pid + a.lay.pitch] - 2.0 * Uc[pid]) + Uc[pid - a.lay.pitch], v);
      }
      if (!RHS && a.use_un) v = fma(a.rk_a, a.Un[c * a.lay.plane + pid], a.rk_b * v);
      out[c] = v;
    }
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) out[c] = RHS ? 0.0 : a.Uin[c * a.lay.plane + pid];
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

// primitives of one cell of the tile box (element e); cells past the array get a uniform state
// (they feed only cells that are not written)
template <int NPL>
__device__ __forceinline__ void put_prims(double* sq, int e, bool in, double r, double mx, double my, double E,
                                          const Gas& g) {
  constexpr int PS = TILE_B * TILE_B;
  double u = 0.0, v = 0.0, p = 1.0, T = 1.0;
  if (in) cons_to_prim(r, mx, my, E, g, u, v, p, T);
  sq[e] = in ? r : 1.0;
  sq[PS + e] = u;
  sq[2 * PS + e] = v;
  sq[3 * PS + e] = p;
  if (NPL == 5) sq[4 * PS + e] = T;
}

// load the conserved tile with halo and convert to primitives in shared memory
template <int NPL>
__device__ __forceinline__ void load_tile(const StageArgs& a, double* sq, int ox, int oy, const Gas& g) {
  const int W = a.lay.nx + 6;
  for (int e = threadIdx.x; e < TILE_B * TILE_B; e += blockDim.x) {
    const int row = e / TILE_B, col = e - row * TILE_B;
    const int gx = ox + col, gy = oy + row;  // padded coordinates
    const bool in = gx < W && gy < a.lay.H;
    const long long s = in ? (long long)gy * a.lay.pitch + gx : 0;
    put_prims<NPL>(sq, e, in, a.Uin[s], a.Uin[a.lay.plane + s], a.Uin[2 * a.lay.plane + s], a.Uin[3 * a.lay.plane + s],
                   g);
  }
}

// ---------------------------------------------------------------------------------------
// TMA staging: one cp.async.bulk.tensor brings the conserved 34 x 34 x 4 box of the padded state
// into shared memory ([plane][row][col]); an mbarrier tracks completion.  Waits are bounded: on
// timeout the block records JS_ERR_TIMEOUT, drains its copy (bounded again) and skips the tile.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// wait for the mbarrier phase `parity` to complete, for at most `budget` SM clock cycles
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, long long budget) {
  const long long t0 = clock64();
  while (true) {
    unsigned ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > budget) return false;
  }
}
__device__ __forceinline__ void tma_box3d(void* dst, const void* map, int x, int y, int z,
                                          unsigned long long* bar, unsigned bytes) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// Stage the tile with TMA and convert it to primitives in place (T in plane 4 when VISC).
// Returns false when the copy did not complete in time (the tile must be skipped).
template <int NPL>
__device__ __forceinline__ bool load_tile_tma(const StageArgs& a, const void* tmap, double* sq, int ox, int oy,
                                              const Gas& g, unsigned long long* bar, unsigned& phase) {
  constexpr int PS = TILE_B * TILE_B;
  constexpr unsigned BYTES = 4u * PS * sizeof(double);
  static_assert(PS * sizeof(double) % 16 == 0 && TILE_B * sizeof(double) % 16 == 0 && TILE * sizeof(double) % 16 == 0,
                "TMA box rows and origins");
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    // the box origin is the tile origin in padded coordinates: x = ox is a multiple of 28 cells
    tma_box3d(sq, tmap, ox, oy, 0, bar, BYTES);
    constexpr long long kBudget = 2000000000LL;  // about one second of SM clock
    bool ok = mbar_wait(bar, phase, kBudget);
    if (!ok) {
      atomicOr(a.err, ERR_TIMEOUT_BIT);
      mbar_wait(bar, phase, kBudget);  // drain the copy in flight before the block moves on
    }
    s_ok = ok ? 1 : 0;
  }
  __syncthreads();
  phase ^= 1u;
  if (!s_ok) return false;
  const int W = a.lay.nx + 6;
  for (int e = threadIdx.x; e < PS; e += blockDim.x) {
    const int row = e / TILE_B, col = e - row * TILE_B;
    put_prims<NPL>(sq, e, ox + col < W && oy + row < a.lay.H, sq[e], sq[PS + e], sq[2 * PS + e], sq[3 * PS + e], g);
  }
  return true;
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

// one tile (bx, by) of one stage; smem holds StageTile::SMEM bytes; whole warps take part
template <bool VISC, bool RHS, bool TMA = false, bool IMG = false>
__device__ __forceinline__ void stage_tile(const StageArgs& a, int bx, int by, double* smem,
                                           const void* tmap = nullptr, unsigned long long* bar = nullptr,
                                           unsigned* phase = nullptr) {
  using S = StageTile<VISC>;
  double* sq = smem;
  double* acc = smem + S::NPL * S::PS;
  const Gas g{a.gamma, a.gm1, a.g1};
  const int tx0 = bx * TILE, ty0 = by * TILE;
  if (TMA) {
    if (!load_tile_tma<S::NPL>(a, tmap, sq, tx0, ty0, g, bar, *phase)) return;
  } else {
    load_tile<S::NPL>(a, sq, tx0, ty0, g);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int k = lane - 2;  // the lane's cell along the line
  // x lines, then y lines (one copy of the code: the strides and planes differ)
#pragma unroll 1
  for (int dir = 0; dir < 2; ++dir) {
    const int lines = dir == 0 ? min(TILE, a.lay.ny - ty0) : min(TILE, a.lay.nx - tx0);
    const int ncell = dir == 0 ? min(TILE, a.lay.nx - tx0) : min(TILE, a.lay.ny - ty0);
    const int st = dir == 0 ? 1 : TILE_B, ts = dir == 0 ? TILE_B : 1;
    const ViscC vc = dir == 0 ? a.vx : a.vy;
    const double cn = dir == 0 ? a.cx : a.cy;
#pragma unroll 1
    for (int ln = warp; ln < lines; ln += nwarp) {
      const double* q = sq + (ln + 3) * ts + (k + 3) * st;
      double dF[4];
      const int gk = (dir == 0 ? tx0 : ty0) + k, gl = (dir == 0 ? ty0 : tx0) + ln;  // cell and line in the grid
      const bool owner = lane >= 2 && k < ncell;
      if constexpr (IMG) {
        line_fluxes<VISC, true>(q, S::PS, st, ts, dir + 1, g, vc, dF, [&](const double* ql, const double* qr) {
          // face gk + 1; the tile's outer face belongs to the next tile unless it is the line's last
          const int f = gk + 1, n = dir == 0 ? a.lay.nx : a.lay.ny;
          if (lane >= 1 && f <= n && (lane <= 28 || (lane == 29 && f == n))) put_image(a, dir, gl, f, ql, qr);
        });
      } else {
        line_fluxes<VISC, true>(q, S::PS, st, ts, dir + 1, g, vc, dF);
      }
      if (owner && lane < 30) {
        const int tx = dir == 0 ? k : ln, ty = dir == 0 ? ln : k;
        double* t = acc + ty * TILE_A + tx;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          double base;
          if (dir == 0) base = RHS ? 0.0 : a.Uin[c * a.lay.plane + a.lay.idx(tx0 + tx, ty0 + ty)];
          else base = t[c * S::PA];
          t[c * S::PA] = fma(-cn, dF[c], base);
        }
      }
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < TILE * TILE; e += blockDim.x) {
    const int ty = e / TILE, tx = e - ty * TILE;
    const int gi = tx0 + tx, gj = ty0 + ty;
    if (gi >= a.lay.nx || gj >= a.lay.ny) continue;
    double upd[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) upd[c] = acc[c * S::PA + ty * TILE_A + tx];
    const int sc = (ty + 3) * TILE_B + tx + 3;
    finish_cell<RHS>(a, gi, gj, upd, sq[sc], sq[3 * S::PS + sc]);
  }
}

}  // namespace js
