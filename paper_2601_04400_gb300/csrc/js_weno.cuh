// WENO5 (Jiang-Shu, eps = 1e-6, power 2; arXiv 2601.04400, Sec. 2) of one cell in integer
// arithmetic (js_wide.cuh says why), cell-centred: both face states of a cell share its three
// smoothness indicators, and an indicator is formed once for the three cells it serves.
//
// The differences d_{j+1/2} = q_{j+1} - q_j and the two final q + c/6 stay FP64 (3 instructions a
// cell, variable and direction, where the whole evaluation took 48); what lies between works on
// 58- to 64-bit mantissas with explicit exponents:
//   * the differences are brought to the largest one's exponent (of the pair for an indicator, of
//     the stencil for the candidate corrections): absolute error 2^-59 of the largest;
//   * indicators, their products and squares are normalised or leave 60 bits; the weights are
//     brought to a common scale on which their sum has 60 to 62 bits;
//   * the quotient takes a 58-bit reciprocal and is rounded to 53 bits at the end.
// The face state's error is that of its final rounding plus about 2^-57 of the largest
// difference: at or below the FP64 sequence's on smooth, noisy and discontinuous data alike, as
// long as the largest difference of the stencil is below 16 |q|.  Where it is not (density or
// pressure on the low side of a jump of 16 or more; velocities pass through zero and are measured
// against the stencil's largest instead) and for differences above 2^477 or not finite, the
// caller takes the FP64 sequence (weno_plain).
#pragma once
#include "js_wide.cuh"

namespace js {

// a first difference d as m 2^(e - 1081): |m| in [2^58, 2^59), or 0
struct Fx {
  s64 m;
  s32 e;
};
JS_HD Fx fx_of(double d) {
  const u64 b = dbits(d);
  const s32 e = expo(d);
  const u64 M = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 6;
  const u64 s = (u64)(s64)((s32)hi32(b) >> 31);
  return Fx{e == 0 ? 0 : (s64)((M ^ s) - s), e};
}

// three times a smoothness indicator, 3 (4 beta_k + 4 eps) = m 2^(x - 2100), 2^63 <= m < 2^64
struct Sm {
  u64 m;
  s32 x;
};
JS_HD Sm sm_norm(u64 s, int x2) {
  const int lz = clz64(s);
  return Sm{s << (lz & 63), x2 - lz};
}
JS_HD double sm_double(const Sm& s) { return bitsd(((u64)(u32)(s.x - 1015) << 52) + (s.m >> 11) + ((s.m >> 10) & 1u)); }

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

// c_L = 6 (q_{i+1/2}^L - q_i) (NL) and c_R = 6 (q_{i-1/2}^R - q_i) (NR) of cell i from its four
// differences and three indicators.  With SV also r_L, r_R = 1 over the weights' sums on the
// scale of (3 s_k)^4 (0 where they leave the FP64 range).
template <bool NL, bool NR, bool SV>
JS_HD void weno_corr(const Fx& dm2, const Fx& dm1, const Fx& dp1, const Fx& dp2, const Sm& s0, const Sm& s1,
                     const Sm& s2, int F, double& cL, double& cR, double& rL, double& rR) {
  // weights w_0 = (s1 s2)^2, w_1 = (s0 s2)^2, w_2 = (s0 s1)^2 (proportional to 1/s_k^2): shifted
  // so that the weighted sums 3 w_0 + 6 w_1 + 3 w_2 (at most X 2^36) stay below 2^62
  const u64 p12 = mul_top(s1.m, s2.m), p02 = mul_top(s0.m, s2.m), p01 = mul_top(s0.m, s1.m);
  const u64 W0 = sqr_top(p12), W1 = sqr_top(p02), W2 = sqr_top(p01);
  const int xm = imin(imin(s0.x, s1.x), s2.x);
  const int n0 = 2 * (s0.x - xm), n1 = 2 * (s1.x - xm), n2 = 2 * (s2.x - xm);
  const u32 X = 3u * (shr32(hi32(W0), n0 + 4) + shr32(hi32(W2), n2 + 4) + 2u * shr32(hi32(W1), n1 + 4) + 4u);
  const int up = 6 - clz32(X);
  const s64 w0 = (s64)shr(W0, n0 + up), w1 = (s64)shr(W1, n1 + up), w2 = (s64)shr(W2, n2 + up);
  const s64 w6 = 6 * w1;
  // differences on the scale of the largest
  const s64 a = sar(dm2.m, F - dm2.e), b = sar(dm1.m, F - dm1.e), c = sar(dp1.m, F - dp1.e), d = sar(dp2.m, F - dp2.e);
  const Limb l6 = limbs(w6);
  const int K = SV ? 2 * (s0.x + s1.x + s2.x) - 2 * xm + up - 8208 : 0;
  if (NL) {  // linear weights 1 : 6 : 3
    const s64 w2_3 = 3 * w2;
    const u64 den = (u64)(w0 + w6 + w2_3);
    const s64 num = mul62(limbs(w0), limbs(5 * b - 2 * a)) + mul62(l6, limbs(b + 2 * c)) +
                    mul62(limbs(w2_3), limbs(4 * c - d));
    const int lz = clz64(den);
    const u64 r = recip_top(den << lz);
    cL = fix_to_double(mul62(limbs(num), limbs((s64)r)), F + lz + 4);
    if (SV) {
      const int be = 959 + lz - K;
      rL = (be < 1 || be > 2046) ? 0.0 : pack62(r, be);
    }
  }
  if (NR) {  // 3 : 6 : 1
    const s64 w0_3 = 3 * w0;
    const u64 den = (u64)(w0_3 + w6 + w2);
    const s64 num = mul62(limbs(w0_3), limbs(a - 4 * b)) + mul62(l6, limbs(-2 * b - c)) +
                    mul62(limbs(w2), limbs(2 * d - 5 * c));
    const int lz = clz64(den);
    const u64 r = recip_top(den << lz);
    cR = fix_to_double(mul62(limbs(num), limbs((s64)r)), F + lz + 4);
    if (SV) {
      const int be = 959 + lz - K;
      rR = (be < 1 || be > 2046) ? 0.0 : pack62(r, be);
    }
  }
}

}  // namespace js
