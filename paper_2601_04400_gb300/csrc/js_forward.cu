// Forward kernels of the FP64 finite-volume step (arXiv 2601.04400, Sec. 2):
//   bc_fill      domain halos (transmissive / reflective / periodic / inflow), 3 deep
//   ib_fill      ghost-cell immersed boundary: slip-wall mirror of the bilinear image-point
//                interpolation of fluid cells (Sec. 2, Fig. 1(c))
//   stage        two kernels per Runge-Kutta stage: lines (primitives, WENO5, HLLC, viscous flux:
//                flux differences of the x and y lines) and cells (divergence, RK combination)
//   stage1d      the same along a single line (ny == 1)
//   cfl_reduce   maximum wave speed and minimum density (bit-exact IEEE arithmetic)
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>

#include "js_device.cuh"
#include "js_internal.h"
#include "js_fill.cuh"
#include "js_stage.cuh"

namespace js {

// =======================================================================================
// domain halo
// =======================================================================================
__global__ void bc_fill_kernel(double* __restrict__ U, Lay lay, BcArgs bc) {
  pdl_enter();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < halo_count(lay)) bc_fill_one(U, lay, bc, t);
}

// =======================================================================================
// immersed-boundary ghost states
// =======================================================================================
__global__ void ib_fill_kernel(double* __restrict__ U, Lay lay, IbArgs ib, double gamma, int wall) {
  pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < 4 * ib.n) ib_fill_one(U, lay, ib, gamma, wall, t);
}

// =======================================================================================
// layout conversion
// =======================================================================================
// a thread per cell, its four planes side by side: bound by memory (2048x1024: 19 us, 7.1 TB/s; a thread
// per value, with 64-bit divisions for its place, took 34)
__global__ void __launch_bounds__(256) pack_kernel(const double* __restrict__ U, double* __restrict__ P, Lay lay) {
  pdl_enter();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= lay.nx) return;
  const long long n = (long long)lay.nx * lay.ny;
  for (int j = blockIdx.y; j < lay.ny; j += gridDim.y) {
    const long long o = (long long)j * lay.nx + i, p = lay.idx(i, j);
    double v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = U[c * n + o];
#pragma unroll
    for (int c = 0; c < 4; ++c) P[c * lay.plane + p] = v[c];
  }
}

__global__ void __launch_bounds__(256) unpack_kernel(const double* __restrict__ P, double* __restrict__ U, Lay lay) {
  pdl_enter();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= lay.nx) return;
  const long long n = (long long)lay.nx * lay.ny;
  for (int j = blockIdx.y; j < lay.ny; j += gridDim.y) {
    const long long o = (long long)j * lay.nx + i, p = lay.idx(i, j);
    double v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = P[c * lay.plane + p];
#pragma unroll
    for (int c = 0; c < 4; ++c) U[c * n + o] = v[c];
  }
}

// row blocks of a [4][ny][nx] state for the halo exchange of a y-decomposed grid
__global__ void rows_pack_kernel(double* __restrict__ U, long long plane, long long off, long long m,
                                 double* __restrict__ buf, int zero) {
  pdl_enter();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * m) return;
  const long long k = (t / m) * plane + off + t % m;
  buf[t] = U[k];
  if (zero) U[k] = 0.0;
}

__global__ void rows_unpack_kernel(double* __restrict__ U, long long plane, long long off, long long m,
                                   const double* __restrict__ buf, int add) {
  pdl_enter();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * m) return;
  const long long k = (t / m) * plane + off + t % m;
  U[k] = add ? U[k] + buf[t] : buf[t];
}

__global__ void prim_to_cons_kernel(const double* W, double* U, long long n, double g1) {
  pdl_enter();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double r = W[t], u = W[n + t], v = W[2 * n + t], p = W[3 * n + t];
  U[t] = r;
  U[n + t] = r * u;
  U[2 * n + t] = r * v;
  U[3 * n + t] = fma(0.5 * r, fma(u, u, v * v), p * g1);
}

// =======================================================================================
// CFL reduction: rate = (|u| + a)/dx [+ (|v| + a)/dy] and rho over fluid cells, the rate in
// IEEE-rounded intrinsics in the oracle's operation order, so equal states give equal dt.
// Small grids take every cell's IEEE rate in one launch.  On larger ones two passes keep that result
// while taking the IEEE rate of few cells: pass 1 takes every fluid cell's rate in FP32, the exact
// minimum density, the maximum of these approximate rates and each block's maximum; pass 2 takes the
// IEEE rate only in blocks, and of cells, whose approximate rate reaches (1 - CFL_MARGIN) of
// that maximum (once per run of cells with identical states along a row).
// The approximation's relative error is that of FP32 times the pressure's cancellation E/p.  Pass 1
// takes FP32 only where the internal energy is above E/16, FP64 with the fast reciprocal only where
// p > 1e-8 E, and the IEEE rate itself elsewhere (near-vacuum cells, non-physical ones), so every
// pass-1 rate is within CFL_MARGIN/2 of the IEEE rate, the cell of the largest IEEE rate is
// always a pass-2 candidate, and the result is the one-pass IEEE maximum for every state.
// The last block of the last launch turns the maximum into the step size (cfl_finish).
// A non-physical fluid cell has the rate +infinity in both passes (cfl_rate).
// =======================================================================================
// block maximum (thread 0 holds it) and, when rmin != nullptr, block minimum
__device__ __forceinline__ void cfl_block_reduce(double& rate, double* rmin) {
  for (int o = 16; o > 0; o >>= 1) {
    rate = fmax(rate, __shfl_xor_sync(0xffffffffu, rate, o));
    if (rmin) *rmin = fmin(*rmin, __shfl_xor_sync(0xffffffffu, *rmin, o));
  }
  __shared__ double sr[32], sm[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    sr[wid] = rate;
    if (rmin) sm[wid] = *rmin;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    rate = (lane < nw) ? sr[lane] : 0.0;
    if (rmin) *rmin = (lane < nw) ? sm[lane] : __longlong_as_double(0x7ff0000000000000LL);
    for (int o = 16; o > 0; o >>= 1) {
      rate = fmax(rate, __shfl_xor_sync(0xffffffffu, rate, o));
      if (rmin) *rmin = fmin(*rmin, __shfl_xor_sync(0xffffffffu, *rmin, o));
    }
  }
}

// the state the reduction reads: the user layout [4][ny][nx] (PADDED false: cell t at t, planes
// n apart) or a context's padded buffer (cell t = (i, j) at off + j pitch + i, planes `plane` apart)
struct CflSrc {
  const double* U;
  long long plane, off;
  int nx, pitch;
};
template <bool PADDED>
__device__ __forceinline__ long long cfl_at(const CflSrc& q, long long t) {
  return PADDED ? q.off + (t / q.nx) * q.pitch + t % q.nx : t;
}

// Device step size from the CFL reduction in red, with js_max_dt's arithmetic (the same IEEE
// operations in the same order): dt = cfl / rate, capped by the viscous limit
// cfl hmin^2 rho_min / (2 mu lim); clipped to t_end - t when t + dt > t_end (t: running time,
// or nullptr), the step inactive once t reaches t_end or when dt is not a positive number
// (a non-physical state: the error flag is set).  Writes the stage constants dtc and dt_log[k].
// Run by the block whose ticket is the last; it leaves red ready for the next step.
__device__ __forceinline__ void cfl_reset(unsigned long long* red) {
  red[0] = 0ULL;                    // IEEE rate maximum
  red[1] = 0x7ff0000000000000ULL;   // density minimum
  red[2] = 0ULL;                    // approximate rate maximum
  red[3] = 0ULL;                    // tickets
}
__device__ __forceinline__ void cfl_finish(unsigned long long* red, const CflStep& q) {
  if (q.dtc == nullptr) return;
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&red[3], 1ULL) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  const int lane = threadIdx.x;
  const double rate = __longlong_as_double((long long)__ldcg(&red[0]));
  const double rmin = __longlong_as_double((long long)__ldcg(&red[1]));
  double dt = __ddiv_rn(q.cfl, rate);
  if (q.visc) {
    const double dtv = __ddiv_rn(__dmul_rn(__dmul_rn(__dmul_rn(q.cfl, q.hmin), q.hmin), rmin),
                                 __dmul_rn(__dmul_rn(2.0, q.mu), q.lim));
    dt = (dtv < dt) ? dtv : dt;
  }
  bool active = dt > 0.0 && dt < CUDART_INF;
  if (!active && lane == 0) atomicOr(q.err, ERR_NONPHYSICAL_BIT);
  double tc = 0.0;
  if (q.t != nullptr) {
    tc = *q.t;
    if (active && q.t_end > 0.0) {
      if (!(tc < q.t_end)) active = false;
      else if (__dadd_rn(tc, dt) > q.t_end) dt = __dsub_rn(q.t_end, tc);
    }
  }
  if (!active) dt = 0.0;
  __syncwarp();
  if (lane < 4) {  // dt/dx, dt/dy, dt nu/dx^2, dt nu/dy^2
    const double h = (lane & 1) ? q.dy : q.dx;
    q.dtc[lane] = __ddiv_rn(lane < 2 ? dt : __dmul_rn(dt, q.nu), lane < 2 ? h : __dmul_rn(h, h));
  }
  if (lane == 4) {
    if (active && q.t != nullptr) *q.t = __dadd_rn(tc, dt);
    q.dtc[4] = active ? 1.0 : 0.0;
    q.dtc[5] = dt;
    if (q.dt_log) q.dt_log[q.k] = dt;
    cfl_reset(red);
  }
}

__global__ void cfl_init_kernel(unsigned long long* red) {
  pdl_enter();
  cfl_reset(red);
}

// Every cell's IEEE rate, a cell a thread (small grids).
template <bool PADDED>
__global__ void __launch_bounds__(128) cfl_one_kernel(CflSrc q, long long n, int two_d,
                                                      const unsigned char* __restrict__ tag, double gamma, double dx,
                                                      double dy, unsigned long long* __restrict__ red, CflStep st) {
  pdl_enter();
  double rate = 0.0, rmin = __longlong_as_double(0x7ff0000000000000LL);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n && !(tag && tag[t] != 0)) {
    const long long e = cfl_at<PADDED>(q, t);
    rmin = q.U[e];
    rate = cfl_rate(rmin, q.U[q.plane + e], q.U[2 * q.plane + e], q.U[3 * q.plane + e], gamma, dx, dy, two_d != 0);
  }
  rmin = fmin(rmin, __longlong_as_double(0x7ff0000000000000LL));
  cfl_block_reduce(rate, &rmin);
  if (threadIdx.x == 0) {
    atomicMax(&red[0], (unsigned long long)__double_as_longlong(rate));
    atomicMin(&red[1], (unsigned long long)__double_as_longlong(rmin));
  }
  cfl_finish(red, st);
}

// (1024x1024 cells: 19 us; with every rate in FP64 56 us, bound by the FP64 pipe)
template <bool PADDED>
__global__ void cfl_pass1_kernel(CflSrc q, long long n, int two_d,
                                 const unsigned char* __restrict__ tag, double gamma, double dx, double dy,
                                 double idx, double idy, unsigned long long* __restrict__ red,
                                 double* __restrict__ bmax) {
  pdl_enter();
  double rate = 0.0, rmin = __longlong_as_double(0x7ff0000000000000LL);
  const double* __restrict__ U = q.U;
  const long long P = q.plane;
  const CflF cf = cfl_f32(gamma, idx, idy, two_d != 0);
  float rf = 0.0f;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    if (tag && tag[t] != 0) continue;
    const long long e = cfl_at<PADDED>(q, t);
    const double r = U[e];
    cfl_rate_max(r, U[P + e], U[2 * P + e], U[3 * P + e], gamma, dx, dy, idx, idy, cf, two_d != 0, rf, rate);
    rmin = fmin(rmin, r);
  }
  rate = fmax(rate, (double)rf);
  cfl_block_reduce(rate, &rmin);
  if (threadIdx.x == 0) {
    // non-negative doubles order like their bit patterns (a negative density is a non-physical
    // cell, whose infinite rate makes the step size 0 whatever the minimum holds)
    bmax[blockIdx.x] = rate;
    atomicMax(&red[2], (unsigned long long)__double_as_longlong(rate));
    atomicMin(&red[1], (unsigned long long)__double_as_longlong(rmin));
  }
}

// A candidate cell whose left neighbour in its row is a fluid cell with the identical state
// leaves the IEEE rate to that neighbour (also a candidate, in a block that passes the test):
// of a uniform run of cells, only the first takes it.  The threads of a warp hold consecutive
// cells, so the neighbour's state comes from the next lower lane.
template <bool PADDED>
__global__ void cfl_pass2_kernel(CflSrc q, long long n, int nx, int two_d,
                                 const unsigned char* __restrict__ tag, double gamma, double dx, double dy,
                                 double idx, double idy, unsigned long long* __restrict__ red,
                                 const double* __restrict__ bmax, CflStep st) {
  pdl_enter();
  const double thr = __longlong_as_double((long long)red[2]) * (1.0 - CFL_MARGIN);
  if (!(bmax[blockIdx.x] >= thr)) {  // the same for the whole block
    cfl_finish(red, st);
    return;
  }
  const CflF cf = cfl_f32(gamma, idx, idy, two_d != 0);
  const int lane = threadIdx.x & 31;
  const double* __restrict__ U = q.U;
  const long long P = q.plane;
  const long long stride = (long long)gridDim.x * blockDim.x;
  double rate = 0.0;
  for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x - lane); base < n; base += stride) {
    const long long t = base + lane;
    const bool in = t < n;
    bool fl = false;
    double r = 0.0, mx = 0.0, my = 0.0, E = 0.0;
    if (in) {
      fl = !(tag && tag[t] != 0);
      const long long e = cfl_at<PADDED>(q, t);
      r = U[e];
      mx = U[P + e];
      my = U[2 * P + e];
      E = U[3 * P + e];
    }
    double rl = __shfl_up_sync(0xffffffffu, r, 1), mxl = __shfl_up_sync(0xffffffffu, mx, 1);
    double myl = __shfl_up_sync(0xffffffffu, my, 1), El = __shfl_up_sync(0xffffffffu, E, 1);
    bool fll = __shfl_up_sync(0xffffffffu, fl ? 1 : 0, 1) != 0;
    if (lane == 0 && in && t > 0) {
      fll = !(tag && tag[t - 1] != 0);
      const long long e = cfl_at<PADDED>(q, t - 1);
      rl = U[e];
      mxl = U[P + e];
      myl = U[2 * P + e];
      El = U[3 * P + e];
    }
    if (in && fl && cfl_reaches(r, mx, my, E, gamma, dx, dy, idx, idy, cf, two_d != 0, thr)) {
      const bool same = (t % nx != 0) && fll && same_bits(r, rl) && same_bits(mx, mxl) && same_bits(my, myl) &&
                        same_bits(E, El);
      if (!same) rate = fmax(rate, cfl_rate(r, mx, my, E, gamma, dx, dy, two_d != 0));
    }
  }
  cfl_block_reduce(rate, nullptr);
  if (threadIdx.x == 0) atomicMax(&red[0], (unsigned long long)__double_as_longlong(rate));
  cfl_finish(red, st);
}

// the stage constants of a launch: the arguments, or those of the device step size
__device__ __forceinline__ bool stage_constants(const StageArgs& a0, StageArgs& a) {
  a = a0;
  if (a0.dtc == nullptr) return true;
  a.cx = a0.dtc[0];
  a.cy = a0.dtc[1];
  a.avx = a0.dtc[2];
  a.avy = a0.dtc[3];
  return a0.dtc[4] != 0.0;
}

// x line blocks, then y line blocks; B: resident blocks an SM the registers are allotted for
template <bool VISC, bool IMG, int B, bool SPLIT = false>
__global__ void __launch_bounds__(32 * SLINES, B) stage_lines_kernel(StageArgs a, int bx) {
  pdl_enter();
  if (a.dtc != nullptr && a.dtc[4] == 0.0) return;  // an inactive device-sized step
  __shared__ double smem[stage_smem<VISC, SPLIT>() / sizeof(double)];
  const int b = blockIdx.x;
  stage_lines<VISC, IMG, SPLIT>(a, b < bx ? 0 : 1, b < bx ? b : b - bx, smem);
}

template <bool RHS>
__global__ void __launch_bounds__(128) stage_cells_kernel(StageArgs a0) {
  pdl_enter();
  StageArgs a;
  if (!stage_constants(a0, a)) return;
  const int gi = blockIdx.x * 128 + threadIdx.x;
  if (gi >= a.lay.nx) return;
  for (int gj = blockIdx.y; gj < a.lay.ny; gj += gridDim.y) stage_cell<RHS>(a, gi, gj);
}

// one line (ny == 1): four warps per 28 cells, a variable's reconstruction each.  Latency up to some
// 30000 cells (one warp per 28 cells: 200 cells 38 us a step, four 30), equal at 70000 and above.
template <bool VISC, bool RHS>
__global__ void __launch_bounds__(128) stage1d_kernel(StageArgs a0) {
  pdl_enter();
  StageArgs a;
  if (!stage_constants(a0, a)) return;
  constexpr int NPL = VISC ? 5 : 4;
  constexpr int PS = SB;
  __shared__ double sq[NPL * PS + 256];
  const Gas g{a.gamma, a.gm1, a.g1};
  const int tx0 = blockIdx.x * SCHUNK, lane = threadIdx.x & 31;
  const int W = a.lay.nx + 6;
  for (int col = threadIdx.x; col < PS; col += 128) {
    const int gx = tx0 + col;
    const int gc = (gx < W) ? gx : W - 1;
    const double r = a.Uin[gc], mx = a.Uin[a.lay.plane + gc], my = a.Uin[2 * a.lay.plane + gc],
                 E = a.Uin[3 * a.lay.plane + gc];
    double u, v, p, T;
    cons_to_prim(r, mx, my, E, g, u, v, p, T);
    sq[col] = r;
    sq[PS + col] = u;
    sq[2 * PS + col] = v;
    sq[3 * PS + col] = p;
    if (NPL == 5) sq[4 * PS + col] = T;
  }
  __syncthreads();
  const int k = lane - 2, gi = tx0 + k;
  double dF[4];
  if (!line_fluxes<VISC, false>(sq + k + 3, PS, 0, 1, g, a.vx, dF, sq + NPL * PS)) return;
  if (lane < 2 || lane > 29 || gi >= a.lay.nx) return;
  if (!(positive(sq[k + 3]) && positive(sq[3 * PS + k + 3]))) atomicOr(a.err, ERR_NONPHYSICAL_BIT);
  finish_cell<RHS>(a, gi, 0, dF, dF);
}

// =======================================================================================
// launchers
// =======================================================================================
namespace {
// Blocks of eight lines up to which four warps share a line: about one block an SM, where a warp's
// chain of four reconstructions is the time.  Per step, shared and not: 96x64 47 and 61 us, 128x128 66
// and 73; then the chip fills: 200x128 (253 blocks) 85 and 80, 250x190 115 and 100.  With face images (two
// steps, FP32 network): 64x48 249 and 288, 128x128 327 and 331, 200x128 502 and 506, 250x190 592 and 560.
constexpr int SPLIT_BLOCKS = GB300_SMS + 8;
// Resident blocks an SM the registers are allotted for: 4 (64 registers, 32 warps) hides the FP64
// and integer latencies best (2048x1024 viscous step: 4 blocks 2.24 ms, 3 blocks 2.30, 2 blocks
// 2.29; 1024x1024 Euler 1.11, 1.14, 1.14).  Tuning variants 1 and 2 are 3 and 2 blocks; every variant gives the same bits.
template <bool VISC, bool IMG>
cudaError_t launch_lines(const StageArgs& a, int variant, cudaStream_t s) {
  const int bx = stage_blocks(a.lay, 0), n = bx + stage_blocks(a.lay, 1);
  if (n <= SPLIT_BLOCKS && variant != 1 && variant != 2) {
    const int sx = stage_blocks(a.lay, 0, SPLIT_LINES);
    return launch(stage_lines_kernel<VISC, IMG, 2, true>, sx + stage_blocks(a.lay, 1, SPLIT_LINES), 32 * SLINES, 0, s, a,
                  sx);
  }
  if constexpr (!IMG) {
    if (variant == 1 || variant == 2) {
      if (variant == 1) launch(stage_lines_kernel<VISC, IMG, 3>, n, 32 * SLINES, 0, s, a, bx);
      else launch(stage_lines_kernel<VISC, IMG, 2>, n, 32 * SLINES, 0, s, a, bx);
      return cudaGetLastError();
    }
  }
  launch(stage_lines_kernel<VISC, IMG, 4>, n, 32 * SLINES, 0, s, a, bx);
  return cudaGetLastError();
}

template <bool VISC, bool IMG = false>
cudaError_t launch_stage2d(const StageArgs& a, bool rhs, int variant, cudaStream_t s) {
  const cudaError_t e = launch_lines<VISC, IMG>(a, variant, s);
  if (e != cudaSuccess) return e;
  const dim3 grid((a.lay.nx + 127) / 128, a.lay.ny < 65535 ? a.lay.ny : 65535);
  if (rhs) launch(stage_cells_kernel<true>, grid, 128, 0, s, a);
  else launch(stage_cells_kernel<false>, grid, 128, 0, s, a);
  return cudaGetLastError();
}

template <bool VISC, bool RHS>
cudaError_t launch_stage1d(const StageArgs& a, cudaStream_t s) {
  return launch(stage1d_kernel<VISC, RHS>, stage_chunks(a.lay.nx), 128, 0, s, a);
}
}  // namespace

cudaError_t launch_stage_img(const StageArgs& a, bool visc, cudaStream_t s) {
  if (a.lay.ny == 1 || a.img == nullptr) return cudaErrorInvalidValue;
  return visc ? launch_stage2d<true, true>(a, false, 0, s) : launch_stage2d<false, true>(a, false, 0, s);
}

cudaError_t launch_stage(const StageArgs& a, bool visc, bool rhs, int variant, cudaStream_t s) {
  if (a.lay.ny == 1) {
    if (visc) return rhs ? launch_stage1d<true, true>(a, s) : launch_stage1d<true, false>(a, s);
    return rhs ? launch_stage1d<false, true>(a, s) : launch_stage1d<false, false>(a, s);
  }
  return visc ? launch_stage2d<true>(a, rhs, variant, s) : launch_stage2d<false>(a, rhs, variant, s);
}

cudaError_t launch_bc_fill(double* U, const Lay& lay, const BcArgs& bc, cudaStream_t s) {
  const long long n = halo_count(lay);
  const int bs = 256;
  launch(bc_fill_kernel, (unsigned)((n + bs - 1) / bs), bs, 0, s, U, lay, bc);
  return cudaGetLastError();
}

cudaError_t launch_ib_fill(double* U, const Lay& lay, const IbArgs& ib, double gamma, int wall, cudaStream_t s) {
  if (ib.n == 0) return cudaSuccess;
  const int bs = 128;
  launch(ib_fill_kernel, (4 * ib.n + bs - 1) / bs, bs, 0, s, U, lay, ib, gamma, wall);
  return cudaGetLastError();
}

cudaError_t launch_pack(const double* U, double* P, const Lay& lay, cudaStream_t s) {
  return launch(pack_kernel, dim3((lay.nx + 255) / 256, std::min(lay.ny, 65535)), 256, 0, s, U, P, lay);
}

cudaError_t launch_unpack(const double* P, double* U, const Lay& lay, cudaStream_t s) {
  return launch(unpack_kernel, dim3((lay.nx + 255) / 256, std::min(lay.ny, 65535)), 256, 0, s, P, U, lay);
}

cudaError_t launch_rows_pack(double* U, int nx, int ny, int row0, int nrows, double* buf, int zero, cudaStream_t s) {
  const long long m = (long long)nrows * nx;
  if (m == 0) return cudaSuccess;
  launch(rows_pack_kernel, (unsigned)((4 * m + 255) / 256), 256, 0, s, U, (long long)nx * ny, (long long)row0 * nx, m,
                                                                   buf, zero);
  return cudaGetLastError();
}

cudaError_t launch_rows_unpack(double* U, int nx, int ny, int row0, int nrows, const double* buf, int add,
                               cudaStream_t s) {
  const long long m = (long long)nrows * nx;
  if (m == 0) return cudaSuccess;
  launch(rows_unpack_kernel, (unsigned)((4 * m + 255) / 256), 256, 0, s, U, (long long)nx * ny, (long long)row0 * nx,
                                                                     m, buf, add);
  return cudaGetLastError();
}

cudaError_t launch_prim_to_cons(const double* W, double* U, long long n, double gamma, cudaStream_t s) {
  const int bs = 256;
  launch(prim_to_cons_kernel, (unsigned)((n + bs - 1) / bs), bs, 0, s, W, U, n, 1.0 / (gamma - 1.0));
  return cudaGetLastError();
}

cudaError_t launch_cfl_init(unsigned long long* red, cudaStream_t s) {
  launch(cfl_init_kernel, 1, 1, 0, s, red);
  return cudaGetLastError();
}

// Cells up to which every rate is taken in IEEE arithmetic at once: one launch in place of two, each of
// which is latency on such grids.  Four steps of 128x64 cells take 200 us with one launch and 210 with two,
// of 256x128 364 and 367; from there the FP64 pipe decides: 200x200 390 and 388, 256x256 525 and 511,
// 400x320 777 and 741.
constexpr long long CFL_ONE_CELLS = 32768;

namespace {
template <bool PADDED>
void cfl_launches(const CflSrc& q, long long n, const Lay& lay, const unsigned char* tag, double gamma, double dx,
                  double dy, unsigned long long* red, double* bmax, const CflStep& st, cudaStream_t s) {
  const int two_d = lay.ny > 1 ? 1 : 0;
  if (n <= CFL_ONE_CELLS) {
    launch(cfl_one_kernel<PADDED>, (unsigned)((n + 127) / 128), 128, 0, s, q, n, two_d, tag, gamma, dx, dy, red, st);
    return;
  }
  const int bs = 256;
  const unsigned blocks = (unsigned)std::min<long long>((n + bs - 1) / bs, CFL_MAX_BLOCKS);
  // both passes on the same grid: a block of pass 2 visits the cells its pass-1 maximum covers
  launch(cfl_pass1_kernel<PADDED>, blocks, bs, 0, s, q, n, two_d, tag, gamma, dx, dy, 1.0 / dx, 1.0 / dy, red, bmax);
  launch(cfl_pass2_kernel<PADDED>, blocks, bs, 0, s, q, n, lay.nx, two_d, tag, gamma, dx, dy, 1.0 / dx, 1.0 / dy, red,
                                                 bmax, st);
}
}  // namespace

int cfl_launch_count(const Lay& lay) { return (long long)lay.nx * lay.ny <= CFL_ONE_CELLS ? 1 : 2; }

cudaError_t launch_cfl(const double* U, const Lay& lay, const unsigned char* tag, double gamma, double dx, double dy,
                       unsigned long long* red, double* bmax, const CflStep& st, cudaStream_t s, bool padded) {
  const long long n = (long long)lay.nx * lay.ny;
  const CflSrc q{U, padded ? lay.plane : n, padded ? lay.idx(0, 0) : 0, lay.nx, padded ? lay.pitch : lay.nx};
  if (padded) cfl_launches<true>(q, n, lay, tag, gamma, dx, dy, red, bmax, st, s);
  else cfl_launches<false>(q, n, lay, tag, gamma, dx, dy, red, bmax, st, s);
  return cudaGetLastError();
}

}  // namespace js
