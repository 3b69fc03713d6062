"""The integer quotient, square root and product of fp64_int.cuh are the IEEE ones, bit for bit,
whatever the FP32 seed's error within +-2 ulp (host build of the same header)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2212_00370_gb300", "csrc")

SOURCE = r"""
#include "fp64_int.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
using namespace rr::fpi;
static int D;
static float off(float r) {
  for (int i = 0; i < std::abs(D); ++i) r = std::nextafterf(r, D < 0 ? 0.f : 4.f);
  return r;
}
struct Seed {
  static float rcp(float x) { return off((float)(1.0 / (double)x)); }
  static float rsqrt(float x) { return off((float)(1.0 / std::sqrt((double)x))); }
};
static double from(uint64_t u) { double x; std::memcpy(&x, &u, 8); return x; }
static const uint64_t F = (1ull << 52) - 1;
static long bad = 0;
static void check(double got, double want, double a, double b) {
  if (std::memcmp(&got, &want, 8) && bad++ < 5) std::printf("%a %a: %a, not %a\n", a, b, got, want);
}
// mantissas near 0 and 1, one and two set bits, short ones, and random ones
static uint64_t mant(std::mt19937_64& g) {
  const uint64_t f = g() & F;
  switch (g() % 6) {
    case 0: return g() % 64;
    case 1: return F - g() % 64;
    case 2: return ((1ull << (g() % 52)) + g() % 3) & F;
    case 3: return f & ~((1ull << (g() % 52)) - 1);
    default: return f;
  }
}
int main(int, char** v) {
  D = std::atoi(v[1]);
  std::mt19937_64 g(7 + D);
  // every leading mantissa of the divisor and of the radicand, with the rest at its ends
  for (uint64_t t = 0; t < (1u << 23); ++t) {
    const uint64_t low = (t % 3 == 0) ? 0 : (t % 3 == 1) ? (1u << 29) - 1 : g() & ((1u << 29) - 1);
    const double b = from((1023ull << 52) | (t << 29) | low);
    const double a = from((1023ull << 52) | ((t & 1) ? mant(g) : ((t << 29) | low) - (t > 0)));
    check(div_fast<Seed>(a, b), a / b, a, b);
    const double x = from(((1023ull + (t & 1)) << 52) | (t << 29) | low);
    check(sqrt_fast<Seed>(x), std::sqrt(x), x, 0);
  }
  for (long i = 0; i < 3000000; ++i) {
    uint64_t ea = 513 + g() % 1022, eb = 513 + g() % 1022;  // the whole exponent window
    if (i % 64 == 0) { ea = (g() & 1) ? 513 : 1534; eb = (g() & 1) ? 513 : 1534; }
    const double a = from((ea << 52) | mant(g) | (g() & (1ull << 63)));
    const double b = from((eb << 52) | mant(g) | (g() & (1ull << 63)));
    check(div_fast<Seed>(a, b), a / b, a, b);
    // next to a midpoint: q = m + 1/2 units, a = q b rounded to either side
    const double m = from((1023ull << 52) | mant(g)), w = std::fabs(b) * std::ldexp(1.0, -std::ilogb(b));
    const double p = (m + std::ldexp(1.0, -52)) * w;
    const double near[3] = {std::nextafter(p, 0.0), p, std::nextafter(p, 9.0)};
    for (double x : near) check(div_fast<Seed>(x, w), x / w, x, w);
    check(sqrt_fast<Seed>(std::fabs(a)), std::sqrt(std::fabs(a)), a, 0);
    const double c = from(((1023 + (ea + g() % 400 - 713) / 2) << 52) | mant(g) | (g() & (1ull << 63)));
    check(mul_fast(c, m), c * m, c, m);                       // and ties: c m with short mantissas
    check(mul_fast(m, m), m * m, m, m);
    check(mul_fast<true>(i % 2 ? c : 0.0 * c, i % 3 ? m : -0.0), (i % 2 ? c : 0.0 * c) * (i % 3 ? m : -0.0), c, m);
    const double y = from(((897 + g() % 253) << 52) | (i % 2 ? mant(g) : (g() & F) | ((1ull << 29) - 1)) | (g() & (1ull << 63)));
    check(to_float_fast(y), (float)y, y, 0);
    check(to_double_fast((float)y), (double)(float)y, y, 0);
    // comparisons on the bits, with zeros, infinities and NaN of both signs
    const double sp[8] = {0.0, -0.0, INFINITY, -INFINITY, NAN, -NAN, 1.0, 0x1p-1074};
    const double u = i % 3 ? a : sp[g() % 8], w2 = i % 5 ? b : sp[g() % 8], n = std::fabs(w2);
    if (gt_nonneg(u, n) != (u > n) && n == n) check(u, n, 1, 1);
    if (pos(u) != (u > 0.0)) check(u, 0, 2, 2);
    if (mag_gt(u, w2) != (std::fabs(u) > std::fabs(w2))) check(u, w2, 3, 3);
    if (n == n && mag_le(u, n) != (std::fabs(u) <= n)) check(u, n, 4, 4);
    if (below_one(std::fabs(u)) != (std::fabs(u) < 1.0)) check(u, 1, 5, 5);
    const double s = (m + std::ldexp(1.0, -53)) * m;
    check(sqrt_fast<Seed>(s), std::sqrt(s), s, 0);
  }
  std::printf("bad %ld\n", bad);
  return bad != 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fp64_int")
    src = d / "t.cpp"
    src.write_text(SOURCE)
    exe = d / "t"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    return str(exe)


@pytest.mark.parametrize("ulps", [-2, -1, 0, 1, 2])
def test_quotient_and_root_are_correctly_rounded(program, ulps):
    r = subprocess.run([program, str(ulps)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
