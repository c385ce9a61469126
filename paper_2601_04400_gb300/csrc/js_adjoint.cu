// Reverse mode of the FP64 finite-volume stage (gradient chain rule of Sec. 2 applied to
// the discrete operator; the hand-written counterpart of backpropagation through the solver
// step of Fig. 1(d)).
//
// One stage VJP, given the adjoint of the stage output and the filled stage state X:
//   lines     per 28 cells of every x and y line: primitives, WENO5 forward, HLLC and viscous forward
//             and reverse per face with Fbar = (lambda'_right - lambda'_left)/h, lambda' = b dt
//             Ubar_next on fluid cells (0 elsewhere), WENO5 reverse: primitive adjoints
//   cells     Ubar(X) = identity and carry terms + the lines' sum through (dprim/dX)^T (+ nu * lap
//             of lambda'); Ubar_0 += a Ubar_next
//   bcT       transposed halo fill (y sides, then x sides), written as gathers;
//             inflow halos accumulate into the inflow-state gradient
//   ibT       transposed immersed-boundary fill: ghost adjoint -> image-point adjoint ->
//             gathered onto the fluid source cells (CSR built on the host)
// Parameter gradients (gamma, mu, Pr, nu, inflow states) are accumulated in pbar.
// No floating-point atomics: every sum runs in a fixed order (per-warp partials of the
// parameter gradient reduced in a fixed order by one block at the end of the stage), so the
// reverse pass gives the same bits on every run.
// With the neural flux on, its reverse runs first, on primitives and lambda' in memory, and the
// lines add its face-state adjoints to their own.
#include <cuda_runtime.h>

#include <algorithm>

#include "js_adjoint_body.cuh"
#include "js_internal.h"

namespace js {

// =======================================================================================
// per-grid launches
// =======================================================================================
// x line blocks, then y line blocks.  Bound by the FP64 pipe (231 instructions a lane, 65% busy) and by
// latency, with the integer WENO5 forward and reverse beside it (57% of issue slots): 1024x512 viscous
// 710 us at B = 4 blocks an SM.  B: the resident blocks the registers are allotted for (ADJ_THREE_BLOCKS).
template <bool VISC, bool SPLIT, int B>
__global__ void __launch_bounds__(32 * ADJ_LINES, B)
adj_lines_kernel(AdjArgs a, const double* __restrict__ Unext, double bdt, int bx) {
  pdl_enter();
  __shared__ double smem[adj_smem(SPLIT)];
  const int b = blockIdx.x;
  adj_lines<VISC, SPLIT>(a, Unext, bdt, b < bx ? 0 : 1, b < bx ? b : b - bx, smem, b);
}

constexpr int kCellThreads = 128;  // (256: 1.2 blocks an SM at 250x190, 23 us against 18)
template <bool VISC>
__global__ void __launch_bounds__(kCellThreads) adj_cells_kernel(AdjArgs a, const double* __restrict__ Unext,
                                                        double* __restrict__ Uacc, double ra, double rb, double bdt,
                                                        int rhs_mode) {
  pdl_enter();
  double gb = 0.0, nb = 0.0;
  adj_cell<VISC>(a, Unext, Uacc, ra, rb, bdt, rhs_mode, (long long)blockIdx.x * blockDim.x + threadIdx.x, gb, nb);
  block_partials(a.pp, blockIdx.x, gb, 0.0, 0.0, nb);
}

// primitives of every padded cell and lambda' = bdt Unext on fluid cells (the neural flux's reverse)
__global__ void adj_nn_seed_kernel(AdjArgs a, double* __restrict__ Q, const double* __restrict__ Unext, double bdt) {
  pdl_enter();
  const Lay& L = a.lay;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= L.plane) return;
  const int col = (int)(t % L.pitch), row = (int)(t / L.pitch);
  if (col >= L.nx + 6 || row >= L.H) return;
  double u, v, p, T;
  const double r = a.X[t];
  cons_to_prim(r, a.X[L.plane + t], a.X[2 * L.plane + t], a.X[3 * L.plane + t], a.gas, u, v, p, T);
  Q[t] = r;
  Q[L.plane + t] = u;
  Q[2 * L.plane + t] = v;
  Q[3 * L.plane + t] = p;
  const int i = col - 3, j = row - L.gy;
  const bool fluid = i >= 0 && i < L.nx && j >= 0 && j < L.ny && (a.tag == nullptr || a.tag[(long long)j * L.nx + i] == 0);
#pragma unroll
  for (int c = 0; c < 4; ++c) a.lam[c * L.plane + t] = fluid ? bdt * Unext[c * L.plane + t] : 0.0;
}

__global__ void adj_bcT_kernel(AdjArgs a, BcArgs bc, int phase_y, double* inflow_part, int tmax) {
  pdl_enter();
  adj_bcT_one(a, bc, phase_y, inflow_part, tmax, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

// the parameter gradient of one stage: four warps sum the inflow halos, the others the partials.  One
// block's latency (one part after the other, the partials by a tree in shared memory: 11 us)
constexpr int kSumThreads = 512;
__global__ void __launch_bounds__(kSumThreads) adj_sums_kernel(AdjArgs a, BcArgs bc, const double* inflow_part,
                                                               int tmax, const double* inflow_prim,
                                                               const double* __restrict__ pp, long long nslot,
                                                               int inflow) {
  pdl_enter();
  __shared__ double S[4][4], part[kSumThreads / 32][4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < 4) {
    if (inflow) adj_inflow_sums(a, bc, inflow_part, tmax, S);
  } else {
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (long long b = threadIdx.x - 128; b < nslot; b += kSumThreads - 128)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] += pp[4 * b + k];
    const double t = warp_sum4(v[0], v[1], v[2], v[3]);
    if ((lane & 7) == 0) part[warp][lane >> 3] = t;
  }
  __syncthreads();
  if (inflow) adj_inflow_states(a, bc, inflow_prim, S);
  if (warp == 1 && lane < 4) {
    double t = lane == 0 && inflow ? adj_inflow_gamma(a, bc, inflow_prim, S) : 0.0;
    for (int w = 4; w < kSumThreads / 32; ++w) t += part[w][lane];
    a.pbar[lane] += t;
  }
}

__global__ void adj_ib_ghost_kernel(AdjArgs a, IbArgs ib, int wall, double* qIb) {
  pdl_enter();
  double gb = 0.0;
  adj_ib_ghost_one(a, ib, wall, qIb, blockIdx.x * blockDim.x + threadIdx.x, gb);
  warp_partials(a.pp, global_warp(), gb, 0.0, 0.0, 0.0);
}

__global__ void adj_ib_src_kernel(AdjArgs a, IbTArgs tb, const double* qIb) {
  pdl_enter();
  double gb = 0.0;
  adj_ib_src_one(a, tb, qIb, blockIdx.x * blockDim.x + threadIdx.x, gb);
  warp_partials(a.pp, global_warp(), gb, 0.0, 0.0, 0.0);
}

__global__ void adj_unpack_add_kernel(const double* __restrict__ P, const double* __restrict__ P2,
                                      double* __restrict__ U, Lay lay) {
  pdl_enter();
  adj_unpack_add_one(P, P2, U, lay, blockIdx.x * blockDim.x + threadIdx.x);
}

// =======================================================================================
// launchers
// =======================================================================================
namespace {
unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }
unsigned ib_blocks(int n) { return n > 0 ? blocks_for(4LL * n, 128) : 0; }  // a quad of lanes an item
}  // namespace

long long adj_strip_doubles(const Lay& L) { return strip_size(L, 0) + strip_size(L, 1); }

// Four warps share a line in 1D (a block of eight lines would hold one) and up to so many blocks of
// eight lines, some 1.5 an SM, where a warp's chain of four reconstructions forward and back is the
// time.  A reverse step, Euler / viscous with a body, shared and not: 64x64 165 / 200 and 238 / 258 us,
// 128x128 249 / 311 and 278 / 341, 180x128 (227 blocks) 305 / 345 and 329 / 351; then the chip fills:
// 250x190 (440) 449 / 527 and 391 / 425.
constexpr int ADJ_SPLIT_BLOCKS = 3 * GB300_SMS / 2;
namespace {
int line_block(const Lay& L) {  // lines a block
  return L.ny == 1 || adj_blocks(L, 0) + adj_blocks(L, 1) <= ADJ_SPLIT_BLOCKS ? ADJ_SPLIT : ADJ_LINES;
}
}  // namespace

long long adj_ppart_doubles(const Lay& L, int n_ghost, int n_src, long long nn_blocks) {
  // slots: one a line block; cells one a block (per warp in the batched kernels); per warp the
  // neural image reverse (256 threads a block) and IB (128)
  const long long slots = adj_blocks(L, 0, line_block(L)) + adj_blocks(L, 1, line_block(L)) + 8 * nn_blocks + 8 * (long long)blocks_for(L.plane, 256) +
                          4 * (long long)(ib_blocks(n_ghost) + ib_blocks(n_src));
  return 4 * slots;
}

cudaError_t launch_adj_stage(const AdjArgs& a0, const BcArgs& bc, const IbArgs& ib, const IbTArgs& ibt, int wall,
                             const double* Unext, double* Uacc, double ra, double rb, double dt, bool rhs_mode,
                             double* inflow_part, const double* inflow_prim, double* qIb, cudaStream_t s,
                             long long* launches, const NnArgs* nn) {
  AdjArgs a = a0;
  const Lay& L = a.lay;
  long long n = 0;
  cudaError_t e;
  // partials of pbar[0..3]: consecutive slices for the launches that produce them
  double* const pp0 = a0.pbar ? a0.pp : nullptr;
  long long used = 0;
  auto slice = [&](long long slots) {
    double* p = pp0 ? pp0 + 4 * used : nullptr;
    used += slots;
    return p;
  };
  if (nn) {
    // the neural flux: its face-state adjoints join the HLLC ones before the WENO5 reverse
    launch(adj_nn_seed_kernel, blocks_for(L.plane, 256), 256, 0, s, a, const_cast<double*>(a.Q), Unext,
                                                                 rhs_mode ? 1.0 : rb * dt);
    a.pp = slice(8 * nn_image_vjp_blocks(L));
    if ((e = nn_reverse(*nn, a, s)) != cudaSuccess) return e;
    n += nn->w_bar ? 14 : 10;
  } else {
    a.fadj = nullptr;
  }
  const double bdt = rhs_mode ? 1.0 : rb * dt;
  const int nl = line_block(L), bx = adj_blocks(L, 0, nl), nb = bx + adj_blocks(L, 1, nl);
  a.pp = slice(nb);
  if (nl == ADJ_SPLIT) {
    if (a.visc) launch(adj_lines_kernel<true, true, 2>, nb, 32 * ADJ_LINES, 0, s, a, Unext, bdt, bx);
    else launch(adj_lines_kernel<false, true, 2>, nb, 32 * ADJ_LINES, 0, s, a, Unext, bdt, bx);
  } else if (nb <= ADJ_THREE_BLOCKS) {
    if (a.visc) launch(adj_lines_kernel<true, false, 3>, nb, 32 * ADJ_LINES, 0, s, a, Unext, bdt, bx);
    else launch(adj_lines_kernel<false, false, 3>, nb, 32 * ADJ_LINES, 0, s, a, Unext, bdt, bx);
  } else {
    if (a.visc) launch(adj_lines_kernel<true, false, 4>, nb, 32 * ADJ_LINES, 0, s, a, Unext, bdt, bx);
    else launch(adj_lines_kernel<false, false, 4>, nb, 32 * ADJ_LINES, 0, s, a, Unext, bdt, bx);
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const unsigned gp = blocks_for(L.plane, kCellThreads);
  a.pp = slice(gp);
  if (a.visc) launch(adj_cells_kernel<true>, gp, kCellThreads, 0, s, a, Unext, Uacc, ra, rb, bdt, rhs_mode ? 1 : 0);
  else launch(adj_cells_kernel<false>, gp, kCellThreads, 0, s, a, Unext, Uacc, ra, rb, bdt, rhs_mode ? 1 : 0);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  n += 2;
  const bool two_d = L.ny > 1;
  a.pp = nullptr;
  const int tmax = std::max(L.nx + 6, L.ny);
  if (two_d) {
    launch(adj_bcT_kernel, blocks_for(8LL * (L.nx + 6), 128), 128, 0, s, a, bc, 1, inflow_part, tmax);
    ++n;
  }
  launch(adj_bcT_kernel, blocks_for(8LL * L.ny, 128), 128, 0, s, a, bc, 0, inflow_part, tmax);
  ++n;
  if (ib.n > 0) {
    a.pp = slice(4LL * ib_blocks(ib.n));
    launch(adj_ib_ghost_kernel, ib_blocks(ib.n), 128, 0, s, a, ib, wall, qIb);
    if (ibt.nsrc > 0) {
      a.pp = slice(4LL * ib_blocks(ibt.nsrc));
      launch(adj_ib_src_kernel, ib_blocks(ibt.nsrc), 128, 0, s, a, ibt, qIb);
    }
    n += 2;
  }
  if (pp0) {
    const int inflow = bc.kind[0] == 3 || bc.kind[1] == 3 || bc.kind[2] == 3 || bc.kind[3] == 3;
    launch(adj_sums_kernel, 1, kSumThreads, 0, s, a, bc, inflow_part, tmax, inflow_prim, pp0, used, inflow);
    ++n;
  }
  if (launches) *launches += n;
  return cudaGetLastError();
}

cudaError_t launch_adj_unpack(const double* P, const double* P2, double* U, const Lay& lay, cudaStream_t s) {
  launch(adj_unpack_add_kernel, blocks_for((long long)lay.nx * lay.ny, 256), 256, 0, s, P, P2, U, lay);
  return cudaGetLastError();
}

}  // namespace js
