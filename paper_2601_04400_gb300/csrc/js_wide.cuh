// 64-bit integer arithmetic that takes work off the FP64 pipe.
//
// GB300 issues one FP64 warp instruction per SM sub-partition about every 80 cycles (DFMA, DADD,
// DMUL and comparisons alike: 1.6 lanes per clock and SM, measured), while 32-bit integer
// multiply-adds, shifts and additions issue every 2 to 6 cycles on their own pipes and run
// beside it (8 wide multiply-adds per DFMA cost nothing, measured).  The routines here carry 58
// to 64 significant bits in integer registers, so their results are at least as accurate as the
// FP64 sequences they replace, at about a tenth of the time.
//
// Plain C++ on purpose: the same source compiles for the host, where the tests compare it with
// higher-precision arithmetic.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define JS_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define JS_HD inline
#endif

namespace js {

typedef uint32_t u32;
typedef uint64_t u64;
typedef int32_t s32;
typedef int64_t s64;

JS_HD u64 dbits(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
JS_HD double bitsd(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}
JS_HD u32 hi32(u64 x) { return (u32)(x >> 32); }
JS_HD u32 mulhi(u32 a, u32 b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (u32)(((u64)a * b) >> 32);
#endif
}
JS_HD int clz64(u64 x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}
JS_HD int clz32(u32 x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
JS_HD int imin(int a, int b) { return a < b ? a : b; }
JS_HD int imax(int a, int b) { return a > b ? a : b; }
// logical and arithmetic right shifts, any non-negative count
JS_HD u64 shr(u64 x, int n) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));  // counts above 63 give 0
  return r;
#else
  return n > 63 ? 0 : x >> n;
#endif
}
JS_HD u32 shr32(u32 x, int n) {
#ifdef __CUDA_ARCH__
  u32 r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));  // counts above 31 give 0
  return r;
#else
  return n > 31 ? 0 : x >> n;
#endif
}
JS_HD s64 sar(s64 x, int n) {
#ifdef __CUDA_ARCH__
  s64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));  // counts above 63 give the sign
  return r;
#else
  return x >> (n > 63 ? 63 : n);
#endif
}

// (a b) >> 64, at most 2 below the exact value
JS_HD u64 mul_top(u64 a, u64 b) {
  const u32 ah = hi32(a), al = (u32)a, bh = hi32(b), bl = (u32)b;
  return (u64)ah * bh + mulhi(ah, bl) + mulhi(al, bh);
}
// (a a) >> 64, at most 2 below the exact value
JS_HD u64 sqr_top(u64 a) {
  const u32 ah = hi32(a), al = (u32)a;
  return (u64)ah * ah + ((((u64)ah * al)) >> 31);
}

// signed 62-bit numbers |x| < 2^62 in two limbs, x = h 2^31 + l with 0 <= l < 2^31: every
// partial product is one signed 32 x 32 -> 64 multiply-add
struct Limb {
  s32 h;
  s32 l;
};
JS_HD Limb limbs(s64 x) { return Limb{(s32)(x >> 31), (s32)((u32)x & 0x7fffffffu)}; }
// (a b) >> 62 up to one unit (the low limbs' product is dropped)
JS_HD s64 mul62(const Limb& a, const Limb& b) {
  const s64 c = (s64)a.h * b.l + (s64)a.l * b.h;
  return (s64)a.h * b.h + (c >> 31);
}
JS_HD s64 sqr62(const Limb& a) { return (s64)a.h * a.h + (((s64)a.h * a.l) >> 30); }

// 2^125 / n for 2^63 <= n < 2^64, relative error below 2^-58, never 2^62 or more: a 23-bit
// hardware seed y and one cubic step y (1 + e + e^2), e = 1 - n y
JS_HD u64 recip_top(u64 n) {
  const u32 nh = hi32(n), nl = (u32)n;
  float f, y;
  const u32 fb = 0x3f800000u | ((nh >> 8) & 0x7fffffu);
#ifdef __CUDA_ARCH__
  f = __uint_as_float(fb);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const u32 Y = __float2uint_rz(y * 2147483648.0f);
#else
  std::memcpy(&f, &fb, 4);
  y = 1.0f / f;
  const u32 Y = (u32)(y * 2147483648.0f);
#endif
  // n Y / 2^32 = 2^62 (1 - e)
  const s64 E = (s64)((1ull << 62) - ((u64)nh * Y + mulhi(nl, Y)));  // e 2^62, |e| < 2^-21
  const s32 Eh = (s32)(E >> 20);                                    // e 2^42
  const s64 G = E + (((s64)Eh * Eh) >> 22);                         // (e + e^2) 2^62
  // y (1 + g) 2^62 = Y 2^31 + Y G / 2^31
  const s64 g = (s64)(s32)(G >> 32) * (s64)Y * 2 + (s64)(((u64)(u32)G * Y) >> 31);
  const u64 r = ((u64)Y << 31) + (u64)g;
  return r - (r >> 62);  // (n = 2^63 exactly would give 2^62)
}

// 2^61 / sqrt(n / 2^64) for 2^62 <= n < 2^64, relative error below 2^-57, never above 2^62 - 1:
// hardware seed y, then y (1 + e/2 + 3 e^2/8), e = 1 - (n / 2^64) y^2
JS_HD u64 rsqrt_top(u64 n) {
  const u32 nh = hi32(n);
  float f, y;
#ifdef __CUDA_ARCH__
  f = __uint2float_rz(nh) * 2.3283064365386963e-10f;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const u32 Y = __float2uint_rz(y * 1073741824.0f);
#else
  f = (float)(nh >> 8) * 5.9604644775390625e-08f;
  y = 1.0f / std::sqrt(f);
  const u32 Y = (u32)(y * 1073741824.0f);
#endif
  const s64 E = (s64)((1ull << 61) - mul_top(n, ((u64)Y * Y) << 1));  // e 2^61, |e| < 2^-20
  const s32 Eh = (s32)(E >> 20);                                      // e 2^41
  const s64 G = (E >> 1) + ((3 * ((s64)Eh * Eh)) >> 24);              // (e/2 + 3 e^2/8) 2^61
  // y (1 + g) 2^61 = Y 2^31 + Y G / 2^30
  const s64 g = (s64)(s32)(G >> 32) * (s64)Y * 4 + (s64)(((u64)(u32)G * Y) >> 30);
  const u64 r = ((u64)Y << 31) + (u64)g;
  return r - (r >> 62);
}

// mantissa of a normal double as 2^63 <= n < 2^64, value n 2^(e - 1086) for the biased exponent e
JS_HD u64 mant64(double x) { return (dbits(x) << 11) | 0x8000000000000000ull; }
JS_HD int expo(double x) { return (int)((hi32(dbits(x)) >> 20) & 0x7ffu); }
// positive double from a mantissa 2^61 <= r < 2^62 and the biased exponent of its leading bit
JS_HD double pack62(u64 r, int be) { return bitsd(((u64)(u32)(be - 1) << 52) + (r >> 9) + ((r >> 8) & 1u)); }

// 1/x (rounded from about 58 bits) for a normal x whose reciprocal is normal: biased exponents
// 1 .. 2044
JS_HD double recip_wide(double x) {
  const double r = pack62(recip_top(mant64(x)), 2045 - expo(x));
  return bitsd(dbits(r) | (dbits(x) & 0x8000000000000000ull));
}
// a/b (rounded from about 57 bits, so within 0.53 ulp) for a normal or zero a and a normal b, rb =
// recip_top(mant64(b)), their quotient normal: biased exponents ea - eb in -1020 .. 1020
JS_HD double quot_wide(double a, double b, u64 rb) {
  const u64 q = mul_top(mant64(a), rb);  // a/b = q 2^(ea - eb - 61), 2^60 <= q < 2^62
  const int lz = clz32(hi32(q));
  const u64 m = q << lz;
  const u64 v = ((u64)(u32)(expo(a) - expo(b) + 1024 - lz) << 52) + (m >> 11) + ((m >> 10) & 1u);
  const u64 sign = (dbits(a) ^ dbits(b)) & 0x8000000000000000ull;
  return bitsd(expo(a) == 0 ? sign : v | sign);
}
// 1/sqrt(x) (rounded from about 57 bits) for a positive normal x
JS_HD double rsqrt_wide(double x) {
  // x = (n / 2^64) 2^(2h), n / 2^64 in [1/4, 1)
  const int e = expo(x) - 1022, odd = e & 1;
  return pack62(rsqrt_top(mant64(x) >> odd), 1023 - ((e + odd) >> 1));
}

// sqrt(g p / r) (rounded from about 57 bits) for positive normal g, p, r: g p and its product with
// 1/sqrt(g p r), all in 64-bit mantissas
JS_HD double sound_wide(double g, double p, double r) {
  const int e = expo(g) + expo(p);
  const u64 gp = mul_top(mant64(g), mant64(p));  // g p = gp 2^(e - 2108)
  const u64 z = mul_top(gp, mant64(r));          // g p r = z 2^(e + e_r - 3130)
  const int lz = clz32(hi32(z));
  const int X = e + expo(r) - 3066 - lz, odd = X & 1;  // g p r = (n / 2^64) 2^X, X even after the shift
  const u64 A = mul_top(gp, rsqrt_top((z << lz) >> odd) << 2);
  const int l2 = clz32(hi32(A));
  const u64 m = A << l2;
  const int be = e - 1021 - l2 - ((X + odd) >> 1);
  return bitsd(((u64)(u32)(be - 1) << 52) + (m >> 11) + ((m >> 10) & 1u));
}

// a signed fixed-point value c 2^(e - 1086) as a double (rounded at 53 bits):
// c / 2^63 in [1/2, 1) has the biased exponent e.  Results below the normal range are subnormal.
// c is the floor of the value meant (right shifts brought it there), so a negative one's magnitude is
// -c - 1 and a fraction: the complement rounds it as a positive value's floor does.
JS_HD double fix_to_double(s64 c, int e) {
  const s64 sg = c >> 63;
  u64 m = (u64)(c ^ sg);
  const int lz = clz64(m);
  m <<= (lz & 63);
  const int be = e - lz;  // biased exponent of the leading bit
  m = shr(m, imax(1 - be, 0));
  // the leading bit adds 1 to the exponent
  const u64 v = ((u64)(u32)imax(be - 1, 0) << 52) + (m >> 11) + ((m >> 10) & 1u);
  return c == 0 ? 0.0 : bitsd(v | ((u64)sg & 0x8000000000000000ull));
}

}  // namespace js
