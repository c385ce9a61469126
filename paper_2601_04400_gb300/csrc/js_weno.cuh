// WENO5 (Jiang-Shu, eps = 1e-6, power 2; arXiv 2601.04400, Sec. 2) of one cell in integer
// arithmetic (js_wide.cuh says why), cell-centred: both face states of a cell share its three
// smoothness indicators, and an indicator is formed once for the three cells it serves.
//
// Everything from the cell values to the face states (48 FP64 instructions a cell, variable and
// direction) works on 58- to 64-bit mantissas with explicit exponents:
//   * the differences d_{j+1/2} = q_{j+1} - q_j are exact, or to 2^-57 where the values' exponents
//     differ; they are brought to the largest one's exponent (of the pair for an indicator, of the
//     stencil for the candidate corrections): absolute error 2^-59 of the largest;
//   * indicators, their products and squares are normalised or leave 60 bits; the weights are
//     brought to a common scale on which their sum has 60 to 62 bits;
//   * the quotient takes a 58-bit reciprocal; the cell value and a sixth of the quotient are added
//     as integers and the sum is rounded to 53 bits, the only rounding.
// The face state's error is that of its final rounding plus about 2^-59 of the largest difference per
// operation (weno_faces), or of each pair's own where a small value lies beside large differences
// (weno_fits).  In units of 2^-53 of |q| and the weighted sum of the candidates' |terms|
// (the scale of FP64's own error), worst of 300,000 stencils against 128 bits, integer and FP64: values
// near rest beside jumps of 1e-4 to 1e4 7.5 and 11, noise 2.1 and 4.5, smooth zero crossings 1.0 and 4.4,
// differences scattered over 8 decades 3.6 and 9.0.  Differences above 2^477 or not finite take the FP64
// sequence (weno_plain).
#pragma once
#include "js_wide.cuh"

namespace js {

// a cell value as m 2^(e - 1080): |m| in [2^57, 2^58), smaller below the normal range (e = 1 there)
struct Qx {
  s64 m;
  s32 e;
};
JS_HD Qx qx_of(double q) {
  const u64 b = dbits(q);
  const s32 e = expo(q);
  const u64 M = ((b & 0x000fffffffffffffull) | (e == 0 ? 0 : 0x0010000000000000ull)) << 5;
  const u64 s = (u64)(s64)((s32)hi32(b) >> 31);
  return Qx{(s64)((M ^ s) - s), imax(e, 1)};
}
// a first difference as m 2^(e - 1081): |m| in [2^58, 2^59) (e may be negative), or 0 with e = 0; e = 2047 where a value
// is not finite or above 2^477
struct Fx {
  s64 m;
  s32 e;
};
JS_HD Fx fx_of(const Qx& hi, const Qx& lo) {
  const int E = imax(hi.e, lo.e);
  const s64 d = sar(hi.m, E - hi.e) - sar(lo.m, E - lo.e);
  const s64 sg = d >> 63;
  const int up = clz64((u64)((d ^ sg) - sg)) - 5;
  return Fx{(s64)((u64)d << (up & 63)), E > 1500 ? 2047 : d == 0 ? 0 : E + 1 - up};
}

// three times a smoothness indicator, 3 (4 beta_k + 4 eps) = m 2^(x - 2100), 2^63 <= m < 2^64
struct Sm {
  u64 m;
  s32 x;
};
JS_HD Sm sm_norm(u64 s, int x2) {
  const int lz = clz32(hi32(s));  // (never below 2^54)
  return Sm{s << lz, x2 - lz};
}

// 3 (4 eps) 2^76, and the exponent of d at which the indicators hold it at that scale: pairs of
// smaller differences keep the scale, larger ones shift it down
constexpr u64 W_EPS = 906694364710971881ull;
constexpr int W_EMIN = 1012;

// The three indicators that one pair of neighbouring differences a = d_{i-1/2}, b = d_{i+1/2}
// determines: s_1 of cell i, s_0 of cell i + 1 and s_2 of cell i - 1.  With D = b - a, t = a + b:
//   4 beta_1 = 13/3 D^2 + t^2,  4 beta_0, 4 beta_2 = 4 beta_1 + 4 D^2 +- 4 D t.
JS_HD void sm_pair(const Fx& a, const Fx& b, Sm& s1, Sm& s0n, Sm& s2p) {
  const int E = imax(imax(a.e, b.e), W_EMIN);
  const s64 am = sar(a.m, E - a.e), bm = sar(b.m, E - b.e);
  const Limb D = limbs(bm - am), t = limbs(am + bm);
  const u64 D2 = (u64)sqr62(D), t2 = (u64)sqr62(t);
  const s64 h = mul62(D, t);
  const u64 v1 = 13u * D2 + 3u * t2 + shr(W_EPS, 2 * (E - W_EMIN));
  const u64 g = v1 + 12u * D2;
  const u64 h12 = (u64)(12 * h);
  s1 = sm_norm(v1, 2 * E);
  s0n = sm_norm(g + h12, 2 * E);
  s2p = sm_norm(g - h12, 2 * E);
}

// weights of one cell: W_k 2^-n_k proportional to 1/s_k^2, and w_k = W_k >> (n_k + up) on the
// scale on which the weighted sum 3 w_0 + 6 w_1 + 3 w_2 (at most X 2^36) has 60 to 62 bits
struct Wgt {
  u64 W0, W1, W2;
  int n0, n1, n2, up;
  s64 w0, w1, w2;
};
JS_HD Wgt weno_weights(const Sm& s0, const Sm& s1, const Sm& s2) {
  Wgt g;
  const u64 p12 = mul_top(s1.m, s2.m), p02 = mul_top(s0.m, s2.m), p01 = mul_top(s0.m, s1.m);
  g.W0 = sqr_top(p12), g.W1 = sqr_top(p02), g.W2 = sqr_top(p01);
  const int xm = imin(imin(s0.x, s1.x), s2.x);
  g.n0 = 2 * (s0.x - xm), g.n1 = 2 * (s1.x - xm), g.n2 = 2 * (s2.x - xm);
  const u32 X = 3u * (shr32(hi32(g.W0), g.n0 + 4) + shr32(hi32(g.W2), g.n2 + 4) + 2u * shr32(hi32(g.W1), g.n1 + 4) + 4u);
  g.up = 6 - clz32(X);
  g.w0 = (s64)shr(g.W0, g.n0 + g.up), g.w1 = (s64)shr(g.W1, g.n1 + g.up), g.w2 = (s64)shr(g.W2, g.n2 + g.up);
  return g;
}

// Whether the common scale serves a cell of value x whose pairs of neighbouring differences reach the
// exponents EL, EM, ER (left, middle, right; F: the largest difference's).  What is added to the value is held
// to 2^-59 of the largest difference, too coarse where the value is small beside it (by 16 or more) and so is
// the correction: gas near rest beside a jump, where a small pair's stencil carries the result.  A velocity
// passes through zero in smooth flow and noise too; there every pair is large, and with it the correction.
// Differences below 2^-11 leave every weight of order one (epsilon).  Of cells of pure noise one in 2,500 is
// refused.
JS_HD bool weno_fits(const Qx& x, int EL, int EM, int ER, int F) {
  return F <= imax(imax(x.e + 3, W_EMIN), imin(imin(EL, EM), ER) + 4);
}

// q_i + num / (6 den), num on the scale 2^(F - 1081 + 62), as a double
JS_HD double weno_face(const Qx& q0, s64 num, u64 den, int F) {
  const u64 d3 = 3u * den;  // below 2^64
  const int lz = clz32(hi32(d3));
  // C 2^(x - 1080) is the correction, |C| below 2^60
  const s64 C = mul62(limbs(num), limbs((s64)recip_top(d3 << lz)));
  const int x = F + lz - 3;
  const int E = imax(q0.e, x);
  return fix_to_double(sar(q0.m, E - q0.e) + sar(C, E - x), E + 6);
}

// Face states of cell i at i+1/2 (left-biased) and i-1/2 (right-biased) from its value, its four
// differences (F: the largest's exponent) and three indicators.  fits (weno_fits): the weighted sum of the
// candidates on the scale of the largest difference.  Else every candidate is formed on its own pair's scale
// and every product of candidate and weight on its own, so that what a small pair contributes keeps its 58
// bits beside a jump (a branch: on every lane it would take a tenth more instructions; with the rule it costs
// 1% of a step: 1024^2 Euler 2.238 ms for two steps, 2.213 without).
JS_HD void weno_faces(const Qx& q0, const Fx& dm2, const Fx& dm1, const Fx& dp1, const Fx& dp2, const Sm& s0,
                      const Sm& s1, const Sm& s2, int F, double& Lf, double& Rf, bool fits = true) {
  const Wgt g = weno_weights(s0, s1, s2);
  s64 numL, numR;  // linear weights 1 : 6 : 3 and 3 : 6 : 1
  int E;
  if (fits) {
    // differences on the scale of the largest
    const s64 a = sar(dm2.m, F - dm2.e), b = sar(dm1.m, F - dm1.e), c = sar(dp1.m, F - dp1.e), d = sar(dp2.m, F - dp2.e);
    const Limb l6 = limbs(6 * g.w1);
    numL = mul62(limbs(g.w0), limbs(5 * b - 2 * a)) + mul62(l6, limbs(b + 2 * c)) + mul62(limbs(3 * g.w2), limbs(4 * c - d));
    numR = mul62(limbs(3 * g.w0), limbs(a - 4 * b)) + mul62(l6, limbs(-2 * b - c)) + mul62(limbs(g.w2), limbs(2 * d - 5 * c));
    E = F;
  } else {
    const int EL = imax(dm2.e, dm1.e), EM = imax(dm1.e, dp1.e), ER = imax(dp1.e, dp2.e);
    // W_k 2^-n_k = N_k 2^-m_k, N_k in [2^63, 2^64); p_k: the exponents of the products
    const Sm N0 = sm_norm(g.W0, 0), N1 = sm_norm(g.W1, 0), N2 = sm_norm(g.W2, 0);
    const int p0 = EL - g.n0 + N0.x, p1 = EM - g.n1 + N1.x, p2 = ER - g.n2 + N2.x, M = imax(imax(p0, p1), p2);
    const Limb l0 = limbs((s64)(N0.m >> 5)), l1 = limbs((s64)(N1.m >> 5)), l2 = limbs((s64)(N2.m >> 5));
    const s64 a = sar(dm2.m, EL - dm2.e), b = sar(dm1.m, EL - dm1.e);
    numL = sar(mul62(limbs(5 * b - 2 * a), l0), M - p0);
    numR = sar(3 * mul62(limbs(a - 4 * b), l0), M - p0);
    const s64 u = sar(dm1.m, EM - dm1.e), v = sar(dp1.m, EM - dp1.e);
    numL += sar(6 * mul62(limbs(u + 2 * v), l1), M - p1);
    numR += sar(6 * mul62(limbs(-2 * u - v), l1), M - p1);
    const s64 c = sar(dp1.m, ER - dp1.e), d = sar(dp2.m, ER - dp2.e);
    numL += sar(3 * mul62(limbs(4 * c - d), l2), M - p2);
    numR += sar(mul62(limbs(2 * d - 5 * c), l2), M - p2);
    E = M + 5 - g.up;
  }
  const s64 w6 = 6 * g.w1;
  Lf = weno_face(q0, numL, (u64)(g.w0 + w6 + 3 * g.w2), E);
  Rf = weno_face(q0, numR, (u64)(3 * g.w0 + w6 + g.w2), E);
}

// ---------------------------------------------------------------------------------------
// Derivatives of c_L and c_R with respect to the cell's four differences a, b, c, d.
// With the normalised weights om_k, the candidates e_k (c = sum om_k e_k) and sigma_k = 3 s_k:
//   dc/dx = sum_k om_k de_k/dx - 4 sum_k Z_k V_kx,   Z_k = om_k (e_k - c),
//   V_kx = (dsigma_k/dx) / (2 sigma_k).
// Z_k is formed from the pairs, Z_0 = om_0 om_1 (e_0 - e_1) + om_0 om_2 (e_0 - e_2) and so on,
// which keeps it accurate where one weight is nearly 1 and e_k - c nearly 0; the differences of
// candidates are multiples of the third differences T_0 = a - 2 b + c, T_1 = b - 2 c + d.  Every
// factor carries its own exponent to the end and each result is rounded from the scale of its own
// weights, so that the derivatives of 1e-12 and less beside a jump are as accurate as the large ones.
// Errors against 128-bit arithmetic: 1e-16 rms, 4 to 6 times below those of the FP64 formulas; in units
// of 2^-53 of the terms' sum at most 12, FP64 16 (jumps, noise, scattered and smooth stencils).
// ---------------------------------------------------------------------------------------
// half the logarithmic derivatives of one indicator with respect to its pair: V = m 2^(960 + k)
struct Lv {
  s64 a, b;
  s32 k;
};

// sm_pair and the derivatives of its three indicators
JS_HD void sm_pair_grad(const Fx& a, const Fx& b, Sm& s1, Sm& s0n, Sm& s2p, Lv& v1, Lv& v0n, Lv& v2p) {
  sm_pair(a, b, s1, s0n, s2p);
  const int E = imax(imax(a.e, b.e), W_EMIN);
  const s64 p = sar(a.m, E - a.e + 3), q = sar(b.m, E - b.e + 3);
  const Limb r1 = limbs((s64)recip_top(s1.m)), r0 = limbs((s64)recip_top(s0n.m)), r2 = limbs((s64)recip_top(s2p.m));
  v1 = Lv{mul62(limbs(8 * p - 5 * q), r1), mul62(limbs(8 * q - 5 * p), r1), E - s1.x};
  v0n = Lv{mul62(limbs(8 * p - 11 * q), r0), mul62(limbs(20 * q - 11 * p), r0), E - s0n.x};
  v2p = Lv{mul62(limbs(20 * p - 11 * q), r2), mul62(limbs(8 * q - 11 * p), r2), E - s2p.x};
}

// x 2^l with 2^60 <= |x 2^l| < 2^61 (two low bits of x dropped)
struct Nm {
  s64 m;
  s32 l;
};
JS_HD Nm nm_of(s64 x) {
  const int l = clz64((u64)(x ^ (x >> 63)) | 1u) - 3;
  return Nm{(x >> 2) << (l + 2), l};
}
// x 2^-n for n of either sign
JS_HD s64 scale_down(s64 x, int n) { return n >= 0 ? sar(x, n) : (s64)((u64)x << (-n)); }

// what both sides' derivatives share
struct GradCell {
  Wgt g;
  Sm N0, N1, N2;       // W_k normalised
  s64 T0, T1;          // third differences on the scale 2^(F - 1081)
  Nm t0, t1;
  Limb v0a, v0b, v1b, v1c, v2c, v2d;
  int k0, k1, k2, F;
};
JS_HD GradCell grad_cell(const Fx& dm2, const Fx& dm1, const Fx& dp1, const Fx& dp2, const Sm& s0, const Sm& s1,
                         const Sm& s2, const Lv& v0, const Lv& v1, const Lv& v2, int F) {
  GradCell q;
  q.g = weno_weights(s0, s1, s2);
  const s64 a = sar(dm2.m, F - dm2.e), b = sar(dm1.m, F - dm1.e), c = sar(dp1.m, F - dp1.e), d = sar(dp2.m, F - dp2.e);
  q.T0 = c - 2 * b + a, q.T1 = d - 2 * c + b;
  // alone, each on the scale of its own differences
  const int EM = imax(dm1.e, dp1.e), F0 = imax(dm2.e, EM), F1 = imax(EM, dp2.e);
  q.t0 = nm_of(sar(dp1.m, F0 - dp1.e) - 2 * sar(dm1.m, F0 - dm1.e) + sar(dm2.m, F0 - dm2.e));
  q.t1 = nm_of(sar(dp2.m, F1 - dp2.e) - 2 * sar(dp1.m, F1 - dp1.e) + sar(dm1.m, F1 - dm1.e));
  q.t0.l += F - F0, q.t1.l += F - F1;
  q.N0 = sm_norm(q.g.W0, q.g.n0), q.N1 = sm_norm(q.g.W1, q.g.n1), q.N2 = sm_norm(q.g.W2, q.g.n2);
  q.v0a = limbs(v0.a), q.v0b = limbs(v0.b), q.v1b = limbs(v1.a), q.v1c = limbs(v1.b), q.v2c = limbs(v2.a), q.v2d = limbs(v2.b);
  q.k0 = v0.k, q.k1 = v1.k, q.k2 = v2.k, q.F = F;
  return q;
}

// o[0..3] = dc/d(a, b, c, d) of the right-biased (right) or left-biased side.  One code copy for both
// (inlined twice and interleaved they take more registers than two blocks an SM leave).
JS_HD void weno_grad_side(const GradCell& q, bool right, double o[4]) {
  const Wgt& g = q.g;
  const u64 den = (u64)((right ? 3 : 1) * g.w0 + 6 * g.w1 + (right ? 1 : 3) * g.w2);
  const int lz = clz32(hi32(den));
  const u64 r = recip_top(den << lz);
  // products of two weights, with their linear weights' product as 3 or 9 times a power of two
  const u64 r4 = r << 2;
  const u64 q0 = mul_top(q.N0.m, r4), q1 = mul_top(q.N1.m, r4), q2 = mul_top(q.N2.m, r4);
  const u64 P01 = mul_top(q0, q1), P02 = mul_top(q0, q2), P12 = mul_top(q1, q2);
  const s64 K01 = right ? (s64)(9 * (P01 >> 6)) : (s64)(3 * (P01 >> 4)), K02 = (s64)(3 * (P02 >> 4)),
            K12 = right ? (s64)(3 * (P12 >> 4)) : (s64)(9 * (P12 >> 6));
  // e_0 - e_1 = -2 T_0 (left), T_0 (right); e_1 - e_2 = T_1, -2 T_1; e_0 - e_2 their sum
  const Nm t02 = nm_of(right ? q.T0 - 2 * q.T1 : q.T1 - 2 * q.T0);
  const s64 E01 = right ? q.t0.m : -q.t0.m, E12 = right ? -q.t1.m : q.t1.m;
  const int m0 = 2 * g.n0 - q.N0.x, m1 = 2 * g.n1 - q.N1.x, m2 = 2 * g.n2 - q.N2.x;  // n_k + lz_k
  const int f = right ? 1 : 0;
  const int h01 = m0 + m1 + q.t0.l - (2 + f), h02 = m0 + m2 + t02.l, h12 = m1 + m2 + q.t1.l - (3 - f);
  // each Z_k on the scale of its own larger part
  const int nu0 = imin(h01, h02), nu1 = imin(h01, h12), nu2 = imin(h02, h12);
  const s64 z01 = mul62(limbs(K01), limbs(E01)), z02 = mul62(limbs(K02), limbs(t02.m)), z12 = mul62(limbs(K12), limbs(E12));
  const Limb Z0 = limbs(sar(z01, h01 - nu0) + sar(z02, h02 - nu0)), Z1 = limbs(sar(z12, h12 - nu1) - sar(z01, h01 - nu1)),
             Z2 = limbs(-sar(z02, h02 - nu2) - sar(z12, h12 - nu2));
  // om_k = O_k 2^e_k, 2^55 <= O_k < 2^56 (c_k q_k = c_k W_k r / 2^62 on the scale 2^(lz - up - 63 - m_k))
  const int L = lz - g.up - 55;
  const Sm u0 = sm_norm(right ? 3 * (q0 >> 2) : q0, L - m0 + (right ? 2 : 0)), u1 = sm_norm(3 * (q1 >> 2), L - m1 + 3),
           u2 = sm_norm(right ? q2 : 3 * (q2 >> 2), L - m2 + (right ? 0 : 2));
  const s64 O0 = (s64)(u0.m >> 8), O1 = (s64)(u1.m >> 8), O2 = (s64)(u2.m >> 8);
  // 4 Z_k V: Z_k on 2^(4 + 2 lz - 2 up - nu_k + F - 1081), V on 2^(960 + k), the product >> 62
  const int x = 2 * lz - 2 * g.up + q.F - 53, x0 = x - nu0 + q.k0, x1 = x - nu1 + q.k1, x2 = x - nu2 + q.k2;
  // an output's scale is that of its larger weight: |4 Z_k V| stays below 34 om_k, so the sums below 2^63
  const int eb = imax(u0.x, u1.x), ec = imax(u1.x, u2.x);
  const s64 b0 = sar(O0, eb - u0.x), b1 = sar(O1, eb - u1.x), c1 = sar(O1, ec - u1.x), c2 = sar(O2, ec - u2.x);
  o[0] = fix_to_double((right ? O0 : -2 * O0) - scale_down(mul62(Z0, q.v0a), u0.x - x0), u0.x + 1086);
  o[1] = fix_to_double((right ? -4 * b0 - 2 * b1 : 5 * b0 + b1) - scale_down(mul62(Z0, q.v0b), eb - x0) -
                           scale_down(mul62(Z1, q.v1b), eb - x1), eb + 1086);
  o[2] = fix_to_double((right ? -c1 - 5 * c2 : 2 * c1 + 4 * c2) - scale_down(mul62(Z1, q.v1c), ec - x1) -
                           scale_down(mul62(Z2, q.v2c), ec - x2), ec + 1086);
  o[3] = fix_to_double((right ? 2 * O2 : -O2) - scale_down(mul62(Z2, q.v2d), u2.x - x2), u2.x + 1086);
}

}  // namespace js
