"""The straight-code quotients and roots of csrc/exact_arith.cuh not only give
the IEEE bits where they settle an operand, they settle nearly all of them, at
every speed a full-orbit particle can have: a form that always refused would be
right and twice the work.  Bounds: a tie band of 0.0005 units on either side of
a midpoint leaves one operand in a thousand, an integer form what its error
bound leaves."""
import ctypes
import subprocess

import numpy as np
import pytest

from tests.test_exact_arith import CSRC, HERE, _load

CODE = r"""
#include <cstdint>
#include <cstring>
static uint64_t g_move;
static float moved(float y) {            // the seeds' bound: two units of FP32
  int b; std::memcpy(&b, &y, 4);
  g_move = g_move * 6364136223846793005ULL + 1442695040888963407ULL;
  b += (int)((g_move >> 33) % 5) - 2;
  std::memcpy(&y, &b, 4);
  return y;
}
#define XA_SEED(y) moved(y)
#include "exact_arith.cuh"
#include "exact_arith_check.h"
using namespace karl;
static double unit(uint64_t r) { return (double)(r >> 11) * 1.1102230246251565e-16; }
struct Vec { double x, y, z; };
static Vec direction(uint64_t i, double u) {
  const double c = 2 * unit(chk_mix(2 * i)) - 1, a = 6.283185307179586 * unit(chk_mix(2 * i + 1));
  const double s = std::sqrt(1 - c * c);
  return {u * s * std::cos(a), u * s * std::sin(a), u * c};
}
static double one_plus(const Vec& v) {
  volatile double a = v.x * v.x, b = v.y * v.y, c = v.z * v.z, ab = a + b, s = ab + c;
  volatile double x = s * (1.0 / (299792458.0 * 299792458.0)), y = 1.0 + x;
  return y;
}
// of n particles of proper speed u and numerators from num to 2 num (of one
// numerator and speed there are only some hundred quotients): settled[0] roots of gamma^2, [1] quotients
// by gamma, [2] gamma by integers, [3] quotients by it, [4] all of a half
// push's; returns the number of wrong settled ones
extern "C" int rates(double u, long long n, double num0, long long* settled) {
  int bad = 0;
  for (int k = 0; k < 5; ++k) settled[k] = 0;
  for (long long i = 0; i < n; ++i) {
    const Vec v = direction((uint64_t)i, u * (1 + 1e-3 * unit(chk_mix(3 * i))));
    const double y = one_plus(v), g = std::sqrt(y), num = num0 * (1 + unit(chk_mix(5 * i)));
    bool r = true, d = true, gi = true, di = true;
    const double gt = xa_sqrt_one_try(y, r);
    const double qt = xa_div_try(num, g, d);
    const int j = xa_gamma_ulps3(v.x, v.y, v.z, gi);
    const long long jg = xa_bits(g) - XA_ONE;
    const double qi = jg < (1 << 30) ? xa_div_1p_try(num, (int)jg, di) : (di = false, 0.0);
    bad += (r && gt != g) + (d && qt != num / g) + (gi && j != jg) + (di && qi != num / g);
    settled[0] += r; settled[1] += d; settled[2] += gi; settled[3] += di;
    bool p = true;
    const double t = xa_div_try(num, xa_sqrt_one_try(y, p), p), t2 = t * t;
    const double sf = xa_div_try(xa_twice(t), 1.0 + t2, p);
    if (p) bad += sf != 2.0 * t / (1.0 + t2);
    settled[4] += p;
  }
  return bad;
}
// roots of 4^e (1 + 37 k 2^-52) and of numbers just below 4^(e + 1), k < n
extern "C" int roots_near_one(long long n) {
  int bad = 0;
  for (long long k = 0; k < n; ++k)
    for (int e = -3; e <= 3; e += 3) {
      const double a = xa_dbl(XA_ONE + k * 37 + (((long long)2 * e) << 52));
      const double b = xa_dbl(XA_ONE + (2LL << 52) - 1 - k + (((long long)2 * e) << 52));
      bool ok = true;
      const double g = xa_sqrt_one_try(a, ok);
      // past 2^27 a root may lie in the tie band
      bad += ok ? g != std::sqrt(a) : k * 37 < (1LL << 27);
      bad += xa_sqrt(b) != std::sqrt(b);
    }
  return bad;
}
"""
U_SMALL = 8500.0                         # csrc/orbit.cu, U2_SMALL
C = 299792458.0
N = 40_000


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rates")
    src, so = d / "rates.cpp", d / "rates.so"
    src.write_text(CODE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    "-I", HERE, "-o", str(so), str(src)], check=True)
    h = ctypes.CDLL(str(so))
    h.rates.argtypes = [ctypes.c_double, ctypes.c_longlong, ctypes.c_double,
                        ctypes.POINTER(ctypes.c_longlong)]
    h.roots_near_one.argtypes = [ctypes.c_longlong]
    return h


# proper speeds from thermal ions to relativistic electrons, closer around the
# ends of the forms (8500 m/s, j = 2^21 at 9.1 km/s, k = 2^27 at 51.8 km/s,
# gamma - 1 = 8 FP32 units at 4.1e5 m/s)
SPEEDS = [30.0, 1e3, 4e3, 5e3, 6e3, 6.6e3, 7e3, 8.4e3, 9e3, 9.3e3, 1e4, 1.5e4, 1.7e4, 2e4, 4e4, 5.1e4,
          5.3e4, 1e5, 2e5, 3e5, 4e5, 4.2e5, 4.5e5, 1e6, 1e7, 1e8, C, 3e9]


@pytest.mark.parametrize("u", SPEEDS)
@pytest.mark.parametrize("num", [0.05, -0.0123456789, 2.27e-12])
def test_settled_at_every_speed(lib, u, num):
    got = (ctypes.c_longlong * 5)()
    assert lib.rates(u, N, num, got) == 0
    root, quo, gam, quo1, push = [g / N for g in got]
    miss = 0.001 + 6 * (0.001 / N) ** 0.5          # the tie band, and chance
    assert root >= 1 - miss
    assert quo >= 1 - miss
    assert push >= 1 - 3 * miss
    if u <= U_SMALL:
        k = (u * 1.001 / C) ** 2 * 2 ** 52         # x 2^52; its bound is k 2^-27 either way of 2
        p = k * 2 ** -27 + 1e-6
        assert gam >= 1 - p - 6 * (p / N) ** 0.5
        p = 4 * (k / 2 + 2) * 2 ** -30             # 4 j 2^-31 either way of 1
        assert quo1 >= 1 - p - 6 * (p / N) ** 0.5
    if u <= 9.1e3:
        assert quo1 > 0.98


def test_roots_next_to_one_and_four(lib):
    # up to 37 x 4e6 = 1.1 x 2^27
    assert lib.roots_near_one(4_000_000) == 0
