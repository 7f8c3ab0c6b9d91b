// Operand sets and checks of csrc/exact_arith.cuh shared by the host and the
// device test: each function against the IEEE operation, bit for bit.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define CHK __device__ __forceinline__
#else
#define CHK static inline
#endif

CHK uint64_t chk_mix(uint64_t x) {
  x += 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  return x ^ (x >> 31);
}
CHK double chk_from(long long b) { return karl::xa_dbl(b); }

// a double of any bit pattern (kind 0), or a normal one with an exponent in
// [-lim, lim] and a significand that is random, next to 1, or next to 2
CHK double chk_number(uint64_t r, int kind, int lim) {
  if (kind == 0) return chk_from((long long)r);
  const long long e = 1023 + (long long)((r >> 3) % (2 * lim + 1)) - lim;
  long long m = (long long)(chk_mix(r) >> 12);
  if (kind == 2) m &= 4095;
  if (kind == 3) m |= ~4095LL & 0x000fffffffffffffLL;
  return chk_from((e << 52) | m);
}
CHK bool chk_same(double a, double b) {
  return karl::xa_bits(a) == karl::xa_bits(b) || (a != a && b != b);
}
// number of failed checks for operand set i
CHK int chk_one(uint64_t i) {
  using namespace karl;
  const uint64_t r1 = chk_mix(3 * i), r2 = chk_mix(3 * i + 1), r3 = chk_mix(3 * i + 2);
  const int lim = (i & 1) ? 40 : 1000;
  double a = chk_number(r1, (int)(r3 % 5), lim), b = chk_number(r2, (int)(r3 / 5 % 5), lim);
  const double p = chk_number(r2, 1, 40), q = chk_number(r1, 1, 40);
  const int near = (int)(r3 / 25 % 4);
  if (near == 1) { b = p; a = p * q; }                       // quotient near a representable number
  if (near == 2) { b = p; a = chk_from(xa_bits(p * q) + 1); }
  int bad = 0;
  if (!(xa_bits(b) < 0)) bad += !chk_same(xa_div(a, b), xa_ieee_div(a, b));
  double s = near == 1 ? q * q : a;                          // root near a representable number
  if (near == 3) s = chk_from(xa_bits(q * q) - 1);
  bad += !chk_same(xa_sqrt(s), xa_ieee_sqrt(s));
  bad += !chk_same(xa_half(a), a * 0.5);
  bad += !chk_same(xa_twice(a), a * 2.0);
  // 1 + x, its root and quotients by the root, x below 2^-25
  double x = chk_from(((long long)(1023 - 26 - (int)(r3 % 60)) << 52) | (long long)(r1 >> 12));
  if (near == 1) x = (double)(2 * (int)(r2 % 100000) + 1) * 1.1102230246251565e-16;   // ties
  const double y = 1.0 + x;
  const int j = (int)((xa_bits(xa_ieee_sqrt(y)) - XA_ONE));
  bad += !chk_same(xa_div_1p(a, j), xa_ieee_div(a, xa_ieee_sqrt(y)));
  const int jt = (int)(r3 >> 40) >> (r3 & 15);
  bad += !chk_same(xa_div_1p(a, jt), xa_ieee_div(a, chk_from(XA_ONE + jt)));
  {
    // components of a proper velocity, of like and unlike sizes
    double u[3];
    const uint64_t r[3] = {r1, r2, r3};
    for (int c = 0; c < 3; ++c) {
      const int spread = (int)((r3 >> 50) & 7) * 5;
      u[c] = chk_from(((long long)(1023 + 8 - (int)(r[c] % (uint64_t)(1 + spread)) + (int)(r3 % 8)) << 52) |
                      (long long)(chk_mix(r[c]) >> 12));
      if ((r3 >> 44) % 16 == (uint64_t)c) u[c] = 0.0;
      if (r[c] & 1024) u[c] = -u[c];
    }
    volatile double sx = u[0] * u[0], sy = u[1] * u[1], sz = u[2] * u[2];
    volatile double sxy = sx + sy, s3 = sxy + sz;
    volatile double x3 = s3 * (1.0 / (299792458.0 * 299792458.0));
    bool ok = true;
    const int j3 = xa_gamma_ulps3(u[0], u[1], u[2], ok);
    if (ok) bad += xa_bits(xa_ieee_sqrt(1.0 + x3)) - XA_ONE != j3;
  }
  return bad;
}
