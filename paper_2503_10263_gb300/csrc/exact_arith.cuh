// exact_arith.cuh - correctly rounded FP64 quotients, roots and sums with few
// instructions on the FP64 pipe.
//
// GB300 issues a warp's FP64 instruction over 64 cycles of its scheduler's
// share of the pipe, an FP32 or integer one over one or two, and the kernels
// that use these functions keep the FP64 pipe busy while most issue slots are
// free.  Each function gives the bits of the IEEE operation it stands for:
// an FP32 seed, two exact FP64 residuals (one fused multiply-add each) whose
// corrections are formed in FP32 and added to the result's bits as integers,
// and a test of the last correction's distance from a rounding boundary (the
// residual form of P. W. Markstein, "Computation of elementary functions on
// the IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990).  Where the
// test cannot decide, or an operand is outside the range treated here (zero,
// subnormal, negative, infinite, NaN, a quotient outside the normal range),
// the IEEE operation itself is called.
//
// The same source compiles for the host (the seeds are then 1/x and
// 1/sqrt(x)), where the tests compare it with the IEEE operations; the result
// does not depend on the seed's last bits.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define XA_FN __device__ __forceinline__
#else
#define XA_FN static inline
#ifndef XA_SEED
#define XA_SEED(y) (y)        // tests perturb the seeds within their bound
#endif
#endif

namespace karl {

#ifdef __CUDACC__
XA_FN long long xa_bits(double x) { return __double_as_longlong(x); }
XA_FN double xa_dbl(long long b) { return __longlong_as_double(b); }
XA_FN int xa_fbits(float x) { return __float_as_int(x); }
XA_FN float xa_flt(int b) { return __int_as_float(b); }
XA_FN double xa_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
XA_FN float xa_fmul(float a, float b) { return __fmul_rn(a, b); }
XA_FN float xa_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
XA_FN float xa_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
XA_FN int xa_rint(float x) { return __float2int_rn(x); }
XA_FN float xa_float(int n) { return __int2float_rn(n); }
// out of line: taken by one operand in a thousand, and by those outside the
// range treated
static __device__ __noinline__ double xa_ieee_div(double a, double b) { return __ddiv_rn(a, b); }
static __device__ __noinline__ double xa_ieee_sqrt(double a) { return __dsqrt_rn(a); }
#else
XA_FN long long xa_bits(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
XA_FN double xa_dbl(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
XA_FN int xa_fbits(float x) { int b; std::memcpy(&b, &x, 4); return b; }
XA_FN float xa_flt(int b) { float x; std::memcpy(&x, &b, 4); return x; }
XA_FN double xa_fma(double a, double b, double c) { return std::fma(a, b, c); }
XA_FN float xa_fmul(float a, float b) { return a * b; }
XA_FN float xa_rcp(float x) { return XA_SEED(1.0f / x); }
XA_FN float xa_rsqrt(float x) { return XA_SEED((float)(1.0 / std::sqrt((double)x))); }
XA_FN int xa_rint(float x) { return (int)std::nearbyint(x); }
XA_FN float xa_float(int n) { return (float)n; }
XA_FN double xa_ieee_div(double a, double b) { return a / b; }
XA_FN double xa_ieee_sqrt(double a) { return std::sqrt(a); }
#endif

constexpr long long XA_ONE = 0x3ff0000000000000LL;
constexpr long long XA_MANT = 0x000fffffffffffffLL;

// The significand of a double as an FP32 number in [1, 2), truncated.
XA_FN float xa_top24(long long b) {
  return xa_flt(0x3f800000 | ((int)(b >> 29) & 0x7fffff));
}
// x truncated to FP32 on the bits; |x| < 2^127, and 0 below 2^-126.
XA_FN float xa_trunc_f(double x) {
  const long long b = xa_bits(x);
  const int h = (int)(b >> 32);
  const int t = (h & 0x7fffffff) - (896 << 20);              // exponent rebiased
  const int m = t < 0 ? 0 : (t << 3) | (int)((unsigned)b >> 29);
  return xa_flt(m | (h & (int)0x80000000));
}
// An FP32 number in [2^-126, 2^127) as a double.
XA_FN double xa_from_f(float f) {
  return xa_dbl(((long long)xa_fbits(f) << 29) + (896LL << 52));
}

// The last correction (in units of the result's last place) lies within 0.5 of
// the integer it is rounded to; beyond XA_TIE its FP32 error (at most 2^-11 of
// a unit, bounded in xa_div and xa_sqrt) could change which integer is
// nearest.  One operand pair in a thousand goes to the IEEE operation.
constexpr float XA_TIE = 0.4995f;

// a / b for b > 0, correctly rounded.  With significands m_a, m_b in [1, 2):
// the seed r ~ 1/m_b is within 2^-22 (truncated operand 2^-23, rcp.approx
// 1 ulp), the quotient q0 = m_a r within 2^-21.7 (the truncations of a and b
// act against each other); the first residual's FP32 correction (relative
// error 2^-21.2) leaves q1 within 2^-42.9, below 2^10.1 units of the last
// place, and the second correction's error is below 2^-11 units.  q0's
// significand must keep eight FP32 units from its binade's ends, so the
// corrections (four of them at most) stay within it (a power of two over a
// divisor next to one does not).  Two FP64 instructions.
// xa_div_try clears ok instead of calling the IEEE division (its value is then
// meaningless), for straight code with one test for many quotients and roots.
XA_FN double xa_div_try(double a, double b, bool& ok) {
  const long long sa = xa_bits(a) & (long long)0x8000000000000000ULL;
  const long long ba = xa_bits(a) ^ sa, bb = xa_bits(b);
  const int ea = (int)(ba >> 52), eb = (int)(bb >> 52);      // eb negative with the sign bit
  const double ma = xa_dbl((ba & XA_MANT) | XA_ONE), mb = xa_dbl((bb & XA_MANT) | XA_ONE);
  const float r = xa_rcp(xa_top24(bb));
  const float q0f = xa_fmul(xa_top24(ba), r);                // in (0.5, 2)
  const int qm = xa_fbits(q0f) & 0x7fffff;
  // 2^52 or 2^53: units of the last place in q0's binade
  const float unit = xa_fbits(q0f) < 0x3f800000 ? 9007199254740992.0f : 4503599627370496.0f;
  const float ru = xa_fmul(r, unit);
  const double q0 = xa_from_f(q0f);
  const double r0 = xa_fma(-q0, mb, ma);
  const int n0 = xa_rint(xa_fmul(xa_trunc_f(r0), xa_fmul(ru, 0.0625f)));   // units of 16
  const long long b1 = xa_bits(q0) + ((long long)n0 << 4);
  const double r1 = xa_fma(-xa_dbl(b1), mb, ma);
  const float c1 = xa_fmul(xa_trunc_f(r1), ru);
  const int n1 = xa_rint(c1);
  const float off = c1 - xa_float(n1);
  // magnitudes in (2^-500, 2^500): normal, and so is the quotient
  ok = ok && (unsigned)(ea - 523) < 1000u && (unsigned)(eb - 523) < 1000u &&
       (unsigned)(qm - 8) < 0x7fffffu - 16u && off < XA_TIE && off > -XA_TIE;
  return xa_dbl((b1 + n1 + ((long long)(ea - eb) << 52)) | sa);
}
XA_FN double xa_div(double a, double b) {
  bool ok = true;
  const double q = xa_div_try(a, b, ok);
  return ok ? q : xa_ieee_div(a, b);
}

// sqrt(a), correctly rounded; the same scheme with m in [1, 4), a = m 4^k,
// the seed y ~ 1/sqrt(m) (rsqrt.approx, 2^-22.3 with the truncated operand)
// and corrections residual x y/2 (the root's second-order term is in the
// first one's relative error, 2^-20.9; the second one's is below 2^-11 units).
// g0 must keep eight FP32 units from 1 and 2, as in xa_div.  Two FP64
// instructions.
// ONE: roots next to one as well (gamma of a slow particle; the others have no
// use for them, and moving-target collisions were 3 % slower with it).  Those of
// m = 1 + k 2^-52 with k < 2^27 are 1 + floor(k/2) 2^-52 (see xa_gamma_ulps3; odd k
// lie next to a midpoint and the corrections could not tell); all others are
// above 1 + 2^-26, and g0, not let below 1, stays there through both corrections.
template <bool ONE> XA_FN double xa_sqrt_form(double a, bool& ok) {
  const long long ba = xa_bits(a);
  const int e = (int)(ba >> 52);
  const int odd = (e & 1) ^ 1;                               // exponent e - 1023 odd
  const long long bm = (ba & XA_MANT) | ((long long)(1023 + odd) << 52);
  const double m = xa_dbl(bm);
  const float mf = xa_flt((xa_fbits(xa_top24(ba))) + (odd << 23));
  const float y = xa_rsqrt(mf);
  const float g = xa_fmul(mf, y), g0f = ONE ? fmaxf(g, 1.0f) : g;
  const int gm = xa_fbits(g0f) - 0x3f800000;                 // its place in [1, 2)
  const float yu = xa_fmul(y, 2251799813685248.0f);          // y/2 x 2^52
  const double g0 = xa_from_f(g0f);
  const double r0 = xa_fma(-g0, g0, m);
  const int n0 = xa_rint(xa_fmul(xa_trunc_f(r0), xa_fmul(yu, 0.0625f)));
  const long long b1 = xa_bits(g0) + ((long long)n0 << 4);
  const double g1 = xa_dbl(b1);
  const double r1 = xa_fma(-g1, g1, m);
  const float c1 = xa_fmul(xa_trunc_f(r1), yu);
  const int n1 = xa_rint(c1);
  const float off = c1 - xa_float(n1);
  const bool even = off < XA_TIE && off > -XA_TIE;
  const long long k = bm - XA_ONE, exp = (long long)((e - odd - 1023) / 2) << 52;
  const bool near1 = ONE && k < (1LL << 27);
  ok = ok && (unsigned)(e - 523) < 1000u &&
       (near1 || ((ONE ? gm < 0x7fffff - 8 : (unsigned)(gm - 8) < 0x7fffffu - 16u) && even));
  return xa_dbl((near1 ? XA_ONE + (k >> 1) : b1 + n1) + exp);
}
XA_FN double xa_sqrt_try(double a, bool& ok) { return xa_sqrt_form<false>(a, ok); }
XA_FN double xa_sqrt_one_try(double a, bool& ok) { return xa_sqrt_form<true>(a, ok); }
XA_FN double xa_sqrt(double a) {
  bool ok = true;
  const double g = xa_sqrt_try(a, ok);
  return ok ? g : xa_ieee_sqrt(a);
}

// j with sqrt(RN(1 + x)) = 1 + j 2^-52, correctly rounded, for 0 <= x < 2^-25.
// RN(1 + x) = 1 + k 2^-52 with k = x 2^52 rounded to nearest even, and its root
// is, in units of 2^-52, k/2 - d with 0 < d = k^2 2^-55 (1 - ...) < 1/2 (d = 0
// at k = 0): an even k gives k/2, an odd one, just below the midpoint, the
// integer below.  So j = floor(k/2) = floor((x 2^52 + 1/2) / 2), ties included.
// For x = RN(RN(RN(RN(ux^2) + RN(uy^2)) + RN(uz^2)) / c^2), gamma of a proper
// velocity of components below 2^14 m/s, it comes from 30-bit fixed-point
// components: their squares' sum S (components rounded, so off by at most
// fx + fy + fz + 1 <= sqrt(3 S) + 1, a relative error below 2^-28 as S >= 2^58)
// times 2^52 / c^2 gives x 2^52 with the error of S; where twice that (2^-27)
// reaches an integer that floor((x 2^52 + 1/2) / 2) turns on, or a component is
// too large, ok is cleared.  (The FP64 chain's own roundings are below 2^-50.)
// No FP64 instruction, against six for the chain.
XA_FN unsigned long long xa_mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDACC__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
XA_FN int xa_gamma_ulps3(double ux, double uy, double uz, bool& ok) {
  const long long bx = xa_bits(ux), by = xa_bits(uy), bz = xa_bits(uz);
  const int ex = (int)(bx >> 52) & 0x7ff, ey = (int)(by >> 52) & 0x7ff, ez = (int)(bz >> 52) & 0x7ff;
  int em = ex > ey ? ex : ey;
  em = em > ez ? em : ez;
  // components in units of 2^(em - 1023 - 29), below 2^30, rounded
  const unsigned long long fx = ((((unsigned)(bx >> 21) | 0x80000000u) >> (em - ex > 30 ? 31 : em - ex + 1)) + 1) >> 1;
  const unsigned long long fy = ((((unsigned)(by >> 21) | 0x80000000u) >> (em - ey > 30 ? 31 : em - ey + 1)) + 1) >> 1;
  const unsigned long long fz = ((((unsigned)(bz >> 21) | 0x80000000u) >> (em - ez > 30 ? 31 : em - ez + 1)) + 1) >> 1;
  const unsigned long long S = fx * fx + fy * fy + fz * fz;
  // (2^56 / c^2) 2^64, rounded
  const unsigned long long hi = xa_mulhi(S, 0xCD3F69CF4136CC8FULL);
  const int s = 4 - 2 * (em - 1023 - 29);                    // x 2^52 = hi 2^-s
  const unsigned long long A = hi + (1ULL << ((s - 1) & 63)), mask = (2ULL << (s & 63)) - 1;
  const unsigned long long rem = A & mask, err = (hi >> 27) + 16;
  ok = ok && em <= 1036 && s < 61 && rem > err && rem < mask - err;
  return (int)(A >> ((s + 1) & 63));
}

// a / (1 + j 2^-52), correctly rounded, for 0 <= j < 2^21 and a normal a: with
// the significand A = 2^52 a', the quotient is A - w, w = a' j (1 - j 2^-52 +
// ...).  w is taken from the 31 upper fraction bits of a', too low by at most
// j 2^-31 for the others and too high by a' j^2 2^-52 <= 2 j 2^-31 for the
// second order; if it is nearer to a midpoint than 4 j 2^-31, or A - w is not
// in a's binade, ok is cleared.  No FP64 instruction.
XA_FN double xa_div_1p_try(double a, int j, bool& ok) {
  const long long ba = xa_bits(a);
  const unsigned a31 = ((unsigned)(ba >> 21) & 0x7fffffffu) | 0x80000000u;   // a' 2^31
  const unsigned long long w = (unsigned long long)a31 * (unsigned)j + (1u << 30);
  const long long n = (long long)(w >> 31);                  // w rounded
  const unsigned rest = (unsigned)w & 0x7fffffffu, near = 4u * (unsigned)j + 4u;
  const int e = (int)(ba >> 52) & 0x7ff;
  ok = ok && (unsigned)j < (1u << 21) && (j == 0 || rest - near < 0x80000000u - 2 * near) &&
       (ba & XA_MANT) >= n && e > 0 && e < 0x7ff;
  return xa_dbl(ba - n);
}
XA_FN double xa_div_1p(double a, int j) {
  bool ok = true;
  const double q = xa_div_1p_try(a, j, ok);
  return ok ? q : xa_ieee_div(a, xa_dbl(XA_ONE + j));
}

// x / 2 and 2 x on the exponent (exact); operands near the ends of the range
// take the multiplication.
XA_FN double xa_half(double x) {
  const long long b = xa_bits(x);
  const int e = (int)(b >> 52) & 0x7ff;
  return e > 1 && e < 0x7ff ? xa_dbl(b - (1LL << 52)) : x * 0.5;
}
XA_FN double xa_twice(double x) {
  const long long b = xa_bits(x);
  const int e = (int)(b >> 52) & 0x7ff;
  return e > 0 && e < 0x7fe ? xa_dbl(b + (1LL << 52)) : x * 2.0;
}

}  // namespace karl
