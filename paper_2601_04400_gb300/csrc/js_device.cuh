// Device building blocks of the FP64 finite-volume right-hand side (arXiv 2601.04400, Sec. 2).
//
// GB300 has a narrow FP64 pipe (about 1/64 of the FP32 rate) while integer, FP32, MUFU and
// min/max work issue on other units.  Everything here is therefore written to minimise
// FP64 add/mul/fma instructions:
//   * no IEEE division or square root: reciprocals and reciprocal square roots are formed in
//     integer arithmetic beside the FP64 pipe (js_wide.cuh), accurate to half an ulp;
//   * WENO5 runs on the integer pipes (js_weno.cuh); the nonlinear weights use the products of the other stencils'
//     (eps + beta)^2 instead of 1/(eps + beta)^2, so one division per face state remains;
//   * HLLC forms the flux of the upwind side's star state (selected with integer selects),
//     the sound speed in integer arithmetic.
#pragma once
#include <cstdint>

#include "js_weno.cuh"

namespace js {

// ---------------------------------------------------------------------------------------
// padded SoA layout of the state: 4 planes [H][pitch], interior cell (i, j) at
// (j + gy) * pitch + i + 3; gy = 3 in 2D and 0 in 1D (ny == 1).
// ---------------------------------------------------------------------------------------
struct Lay {
  int nx, ny, gy, pitch, H;
  long long plane;
  __host__ __device__ long long idx(int i, int j) const { return (long long)(j + gy) * pitch + (i + 3); }
};

constexpr int ERR_NONPHYSICAL_BIT = 1;
constexpr int ERR_TIMEOUT_BIT = 2;

// ---------------------------------------------------------------------------------------
// FP64 reciprocal / quotient / reciprocal square root that leave the FP64 pipe free
// ---------------------------------------------------------------------------------------
// The cases outside the integer routines' range (zero, subnormal, infinite, NaN; a negative
// square root) take the FP64 forms: MUFU seeds, accurate to about 2^-20 (measured on GB300), and
// one cubic (Halley) step.
static __device__ __noinline__ double recip_plain(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
static __device__ __noinline__ double rsqrt_plain(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}
// 1/x in integer arithmetic (js_wide.cuh), correctly rounded but for one in 2000 arguments
// where the seed and Halley step reached about 1.5 ulp; it takes no FP64 issue slot instead of 3
__device__ __forceinline__ double recip(double x) {
  if ((u32)(expo(x) - 1) >= 2044u) return recip_plain(x);
  return recip_wide(x);
}
// a/b as a * (1/b) (1 FP64 instruction; within 1 ulp)
__device__ __forceinline__ double quot(double a, double b) { return a * recip(b); }
// a/b within 0.53 ulp in integer arithmetic, rb = recip_top(mant64(b)) (formed ahead of a); IEEE division
// outside that routine's range
__device__ __forceinline__ double quot_near(double a, double b, u64 rb) {
  const int ea = expo(a), eb = expo(b);
  const bool out = (u32)(ea - 1) >= 2046u || (u32)(ea - eb + 1020) > 2040u;
  if ((u32)(eb - 1) >= 2046u || (out && (dbits(a) << 1) != 0)) return a / b;
  return quot_wide(a, b, rb);
}
// 1/sqrt(x) likewise (0 instead of 5 FP64 instructions)
__device__ __forceinline__ double rsqrt_nr(double x) {
  const s32 h = (s32)hi32(dbits(x));
  if ((u32)(h - 0x00100000) >= 0x7fe00000u) return rsqrt_plain(x);  // not positive and normal
  return rsqrt_wide(x);
}

// sound speed sqrt(gamma p / r) in integer arithmetic (it took 8 FP64 instructions)
__device__ __forceinline__ double sound(double gamma, double p, double r) {
  const s32 hp = (s32)hi32(dbits(p)), hr = (s32)hi32(dbits(r));
  if ((u32)(hp - 0x00100000) >= 0x7fe00000u || (u32)(hr - 0x00100000) >= 0x7fe00000u) {
    const double gp = gamma * p;
    return gp * rsqrt_plain(gp * r);
  }
  return sound_wide(gamma, p, r);
}

// ---------------------------------------------------------------------------------------
// gas constants of one launch
// ---------------------------------------------------------------------------------------
struct Gas {
  double gamma, gm1, g1;  // gamma, gamma - 1, 1/(gamma - 1)
};

// primitive variables of a conserved state; returns T = p/rho as well
__device__ __forceinline__ void cons_to_prim(double r, double mx, double my, double E, const Gas& g,
                                             double& u, double& v, double& p, double& T) {
  const double ir = recip(r);
  u = mx * ir;
  v = my * ir;
  const double k2 = fma(mx, u, my * v);  // rho (u^2 + v^2)
  p = g.gm1 * fma(-0.5, k2, E);
  T = p * ir;
}

// ---------------------------------------------------------------------------------------
// WENO5 (Jiang-Shu, eps = 1e-6, power 2) on a line, cell-centred.
// For cell i with neighbours q_{i-2..i+2} (Sec. 2: reconstruction of primitive variables):
//   d_{i+1/2} = q_{i+1} - q_i,  D_i = q_{i-1} - 2 q_i + q_{i+1}
//   4 beta_0 = 13/3 D_{i-1}^2 + (D_{i-1} + 2 d_{i-1/2})^2
//   4 beta_1 = 13/3 D_i^2     + (d_{i-1/2} + d_{i+1/2})^2
//   4 beta_2 = 13/3 D_{i+1}^2 + (D_{i+1} - 2 d_{i+1/2})^2
// s_k = 4 beta_k + 4 eps; the weights alpha_k = d_k / s_k^2 are scaled by (s0 s1 s2)^2.
// Candidate values minus q_i, times 6, are two-term combinations of the d's.  weno_lane and
// weno_cell evaluate this in integer arithmetic (js_weno.cuh), weno_plain in FP64.
// ---------------------------------------------------------------------------------------
constexpr double EPS12 = 1.2e-5;  // 3 (4 eps)
constexpr double SIXTH = 1.0 / 6.0;

// Network input of one face (neural flux, Sec. 2.3): the mean of its two WENO5 face states
// (primitive rho, u, v, p in wl / wr; un / ut the planes of the face-normal and tangential
// velocity) in conserved variables of the face frame, normalised by mean and 1/sd per channel,
// in arithmetic R: double for the FP64 network, float for the FP32 and BF16 networks (whose input
// is FP32: the face states are rounded to FP32 first, sparing the FP64 pipe).  One definition for
// every kernel that forms face images, so that they agree bit for bit.
template <class R>
__device__ __forceinline__ void face_image(const double wl[4], const double wr[4], int un, int ut, R g1,
                                           const R mean[4], const R inv_sd[4], R m[4]) {
  const R rL = (R)wl[0], rR = (R)wr[0], nL = (R)wl[un], nR = (R)wr[un], tL = (R)wl[ut], tR = (R)wr[ut];
  const R pL = (R)wl[3], pR = (R)wr[3], h = (R)0.5;
  const R EL = fma(h * rL, fma(nL, nL, tL * tL), pL * g1);
  const R ER = fma(h * rR, fma(nR, nR, tR * tR), pR * g1);
  m[0] = h * (rL + rR);
  m[1] = h * fma(rL, nL, rR * nR);
  m[2] = h * fma(rL, tL, rR * tR);
  m[3] = h * (EL + ER);
#pragma unroll
  for (int k = 0; k < 4; ++k) m[k] = (m[k] - mean[k]) * inv_sd[k];
}

// the FP64 form of one cell: its face states at i+1/2 (left-biased) and i-1/2 (right-biased)
static __device__ __noinline__ double2 weno_plain(double qm2, double qm1, double q0, double q1, double q2) {
  const double dm2 = qm1 - qm2, dm1 = q0 - qm1, dp1 = q1 - q0, dp2 = q2 - q1;
  const double D0 = dm1 - dm2, D1 = dp1 - dm1, D2 = dp2 - dp1;
  const double t0 = fma(2.0, dm1, D0), t1 = dm1 + dp1, t2 = fma(-2.0, dp1, D2);
  const double s0 = fma(13.0 * D0, D0, fma(3.0 * t0, t0, EPS12));
  const double s1 = fma(13.0 * D1, D1, fma(3.0 * t1, t1, EPS12));
  const double s2 = fma(13.0 * D2, D2, fma(3.0 * t2, t2, EPS12));
  const double p01 = s0 * s1, p02 = s0 * s2, p12 = s1 * s2;
  const double w0 = p12 * p12, w1 = p02 * p02, w2 = p01 * p01;  // proportional to 1/s_k^2
  const double w6 = 6.0 * w1, w2_3 = 3.0 * w2, w0_3 = 3.0 * w0;
  // left-biased (linear weights 0.1 : 0.6 : 0.3), right-biased (0.3 : 0.6 : 0.1)
  const double nL = fma(w0, fma(-2.0, dm2, 5.0 * dm1), fma(w6, fma(2.0, dp1, dm1), w2_3 * fma(4.0, dp1, -dp2)));
  const double nR = fma(w0_3, fma(-4.0, dm1, dm2), fma(w6, fma(-2.0, dm1, -dp1), w2 * fma(2.0, dp2, -5.0 * dp1)));
  return make_double2(fma(quot(nL, w0 + w6 + w2_3), SIXTH, q0), fma(quot(nR, w0_3 + w6 + w2), SIXTH, q0));
}

__device__ __forceinline__ Sm shfl_up(const Sm& s) {
  return Sm{(u64)__shfl_up_sync(0xffffffffu, (unsigned long long)s.m, 1), __shfl_up_sync(0xffffffffu, s.x, 1)};
}
__device__ __forceinline__ Sm shfl_down(const Sm& s) {
  return Sm{(u64)__shfl_down_sync(0xffffffffu, (unsigned long long)s.m, 1), __shfl_down_sync(0xffffffffu, s.x, 1)};
}
__device__ __forceinline__ Fx shfl_up(const Fx& d) {
  return Fx{(s64)__shfl_up_sync(0xffffffffu, (long long)d.m, 1), __shfl_up_sync(0xffffffffu, d.e, 1)};
}
__device__ __forceinline__ Fx shfl_down(const Fx& d) {
  return Fx{(s64)__shfl_down_sync(0xffffffffu, (long long)d.m, 1), __shfl_down_sync(0xffffffffu, d.e, 1)};
}

// Face states at i+1/2 (Lf, left-biased) and i-1/2 (Rf, right-biased) of one cell per lane: the
// lanes of a warp hold consecutive cells of a line, q points at the lane's own (q[-st .. st]
// readable; q[-2 st], q[2 st] too in the inner lanes 1..30, where the result is valid).  A lane
// forms the differences on both sides of its cell and the three indicators they determine, and
// takes its s_0, s_2 and outer differences from its neighbours.
__device__ __forceinline__ void weno_lane(const double* q, int st, bool inner, double& Lf, double& Rf) {
  const Qx x = qx_of(q[0]);
  const Fx dm1 = fx_of(x, qx_of(q[-st])), dp1 = fx_of(qx_of(q[st]), x);
  Sm s1, s0n, s2p;
  sm_pair(dm1, dp1, s1, s0n, s2p);
  const Sm s0 = shfl_up(s0n), s2 = shfl_down(s2p);
  const Fx dm2 = shfl_up(dm1), dp2 = shfl_down(dp1);
  const int EL = imax(dm2.e, dm1.e), EM = imax(dm1.e, dp1.e), ER = imax(dp1.e, dp2.e), F = imax(EL, ER);
  if (F > 1500 && inner) {
    const double2 r = weno_plain(q[-2 * st], q[-st], q[0], q[st], q[2 * st]);
    Lf = r.x;
    Rf = r.y;
  } else {
    weno_faces(x, dm2, dm1, dp1, dp2, s0, s1, s2, F, Lf, Rf, weno_fits(x, EL, EM, ER, F));
  }
}

// the same for a single thread (q[-2 st .. 2 st] readable): the same bits
template <class I>
__device__ __forceinline__ void weno_cell(const double* q, I st, double& Lf, double& Rf) {
  const Qx m2 = qx_of(q[-2 * st]), m1 = qx_of(q[-st]), x = qx_of(q[0]), p1 = qx_of(q[st]), p2 = qx_of(q[2 * st]);
  const Fx dm2 = fx_of(m1, m2), dm1 = fx_of(x, m1), dp1 = fx_of(p1, x), dp2 = fx_of(p2, p1);
  Sm s0, s1, s2, u, v;
  sm_pair(dm2, dm1, u, s0, v);
  sm_pair(dp1, dp2, u, v, s2);
  sm_pair(dm1, dp1, s1, u, v);
  const int EL = imax(dm2.e, dm1.e), EM = imax(dm1.e, dp1.e), ER = imax(dp1.e, dp2.e), F = imax(EL, ER);
  if (F > 1500) {
    const double2 r = weno_plain(q[-2 * st], q[-st], q[0], q[st], q[2 * st]);
    Lf = r.x;
    Rf = r.y;
  } else {
    weno_faces(x, dm2, dm1, dp1, dp2, s0, s1, s2, F, Lf, Rf, weno_fits(x, EL, EM, ER, F));
  }
}

// ---------------------------------------------------------------------------------------
// HLLC (Sec. 2) in the face-normal frame.  State (rho, un, ut, p) on each side; returns
// [mass, normal momentum, tangential momentum, energy].  Star-state energy in the
// standard (Toro) form.
//
// Of the upwind side K of the contact (s* > 0: left), with d = s_K - u, m = rho d and the star
// pressure p* = p + m (s* - u), the flux F_K + s_K (U*_K - U_K) equals the flux of the star state
// (the jump relation across s_K), which is formed directly:
//   G = m s*/(s_K - s*),  F = (G, G s* + p*, G u_t, s*/(s_K - s*) (d E - p u + p* s_K)).
// A supersonic face (s_K on the far side of zero) has F = F_K, the same expressions with u in
// the place of s*.  At s* = 0 both sides give (0, p*, 0, 0): the average of the branches that
// sign(0) = 0 asks for is either of them.  31 FP64 instructions a face (15 at s* = 0, where gas
// at rest on both sides always lands) where building the star state and its jump took 69.
// ---------------------------------------------------------------------------------------
// signs and positivity from the bits: an FP64 comparison takes an FP64 issue slot
__device__ __forceinline__ bool sign_clear(double x) { return (s32)hi32(dbits(x)) >= 0; }
// x > 0 (false for NaN)
__device__ __forceinline__ bool positive(double x) { return dbits(x) - 1u < 0x7ff0000000000000ull; }

__device__ __forceinline__ void hllc(double rL, double uL, double vL, double pL, double rR, double uR,
                                     double vR, double pR, const Gas& g, double F[4]) {
  const double aL = sound(g.gamma, pL, rL), aR = sound(g.gamma, pR, rR);
  const double sL = fmin(uL - aL, uR - aR);
  const double sR = fmax(uL + aL, uR + aR);
  // (products that a later sum or difference could be contracted with are rounded on their own:
  // every kernel that inlines this then gives the same bits)
  const double dL = sL - uL, dR = sR - uR;
  const double mL = __dmul_rn(rL, dL), mR = __dmul_rn(rR, dR);
  const double num = fma(-uR, mR, fma(uL, mL, pR - pL));
  const double ss = __dmul_rn(num, recip(mL - mR));
  const bool left = sign_clear(ss);
  const double u = left ? uL : uR, ut = left ? vL : vR, p = left ? pL : pR, s = left ? sL : sR,
               d = left ? dL : dR, m = left ? mL : mR;
  const bool outside = sign_clear(left ? sL : -sR);  // s_L >= 0, s_R <= 0
  const double c = outside ? u : ss;
  const double ps = fma(m, c - u, p);
  if ((dbits(c) << 1) == 0) {  // gas at rest on both sides: nothing but the pressure
    F[0] = F[2] = F[3] = 0.0;
    F[1] = ps;
    return;
  }
  const double w = __dmul_rn(c, recip(s - c));
  const double G = __dmul_rn(m, w);
  // d E = m (u^2 + u_t^2)/2 + d p/(gamma - 1)
  const double dE = fma(0.5 * m, fma(u, u, ut * ut), g.g1 * (d * p));
  F[0] = G;
  F[1] = fma(G, c, ps);
  F[2] = __dmul_rn(G, ut);
  F[3] = __dmul_rn(w, fma(ps, s, fma(-p, u, dE)));
}

// ---------------------------------------------------------------------------------------
// Navier-Stokes viscous and heat flux through a face (constant mu, Stokes hypothesis,
// R = 1).  Normal derivatives by two-point differences, tangential ones by the mean of the
// central differences of the two adjacent cells.  Constants (per face orientation):
//   c43n = 4/3 mu / h_n, c23t = 2/3 mu / (4 h_t), cn = mu / h_n, ct = mu / (4 h_t),
//   ck = kappa / h_n with kappa = mu gamma / ((gamma - 1) Pr).
// ---------------------------------------------------------------------------------------
struct ViscC {
  double c43n, c23t, cn, ct, ck;
};

}  // namespace js
