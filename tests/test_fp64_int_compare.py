"""The comparisons and windows on the bits (fp64_int.cuh) agree with the FP64 ones for every
pair of zeros, the smallest and largest numbers, powers of two and their neighbours, infinities
and NaN of both signs, equal operands among them (host build of the same header)."""
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
#include <vector>
using namespace rr::fpi;
static long bad = 0, n = 0;
static void check(const char* what, bool got, bool want, double x, double y) {
  ++n;
  if (got != want && bad++ < 20) std::printf("%s(%a, %a): %d\n", what, x, y, (int)got);
}
int main() {
  std::vector<double> v;
  for (double x : {0.0, 0x1p-1074, 0x1p-1022, 0x1p-126, 0x1p-80, 0.5, 1.0, 3.0, 0x1p80, 0x1p127,
                   0x1p1023, (double)INFINITY, (double)NAN})
    for (double s : {1.0, -1.0})
      for (double y : {x, std::nextafter(x, 0.0), std::nextafter(x, (double)INFINITY)}) v.push_back(std::copysign(y, s));
  for (double x : v) {
    check("pos", pos(x), x > 0.0, x, 0);
    if (!(x < 0.0) && !(std::signbit(x) && x == 0.0)) check("below_one", below_one(x), x < 1.0, x, 1);
    for (int lo : {-200, -80, 0, 1}) {
      const double a = std::fabs(x), l = std::ldexp(1.0, lo), h = std::ldexp(1.0, lo + 80);
      check("in_window", in_window(x, 1023 + lo, 80), a >= l && a < h, x, l);
      check("in_window_or_zero", in_window_or_zero(x, 1023 + lo, 80), (a >= l && a < h) || a == 0.0, x, l);
    }
    for (double y : v) {
      const double a = std::fabs(y);
      check("mag_gt", mag_gt(x, y), std::fabs(x) > a, x, y);
      if (a != a) continue;  // the second operand of the others is a number >= 0
      check("gt_nonneg", gt_nonneg(x, a), x > a, x, a);
      check("mag_le", mag_le(x, a), std::fabs(x) <= a, x, a);
    }
  }
  std::printf("%ld checks, %ld bad\n", n, bad);
  return bad != 0 || n < 10000;
}
"""


def test_comparisons_on_the_bits(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
