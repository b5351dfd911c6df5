"""rcp64 and rsqrt64 (dg_common.cuh) with the approximate instructions at the ends of
their documented error: rcp.approx.ftz.f32 within 1 unit in the last place,
rsqrt.approx.ftz.f32 within 2^-22.9, up to 2 units where the result is just above a
power of two. The header's host stand-ins round correctly; here they are moved by -2
to 2 units (rcp: -1 to 1). Significands near the ends of [1, 4), where an
approximation can fall below 0.5, and all over it. Bound: 0.52 units in the last
place of the FP64 result, as for exact approximations (the iteration's error term is
the cube of theirs, below 2^-62)."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cmath>
static int g_move = 0;
static float moved(float y, int most) {
  const int n = g_move < -most ? -most : g_move > most ? most : g_move;
  for (int i = 0; i < (n < 0 ? -n : n); ++i) y = std::nextafter(y, n < 0 ? 0.f : 8.f);
  return y;
}
#include "roots.cuh"
#include <random>
using namespace dg;
static double ulps(double y, long double t) {
  const double a = std::fabs((double)t);
  return (double)(fabsl((long double)y - t) / (long double)(std::nextafter(a, INFINITY) - a));
}
int main() {
  std::mt19937_64 g(2);
  double e[2] = {0, 0};
  for (g_move = -2; g_move <= 2; ++g_move)
    for (long i = 0; i < 600000; ++i) {
      unsigned long long b = g() & 0xfffffffffffffull;
      if (i % 3 == 0) b >>= 8 + i % 41;                            // just above a power of two
      if (i % 3 == 1) b = 0xfffffffffffffull - (b >> (8 + i % 41));  // just below
      b |= (unsigned long long)(1022 + i % 4) << 52;
      double x;
      std::memcpy(&x, &b, 8);
      e[0] = std::max(e[0], ulps(rcp64(x), 1.0L / x));
      e[1] = std::max(e[1], ulps(rsqrt64(x), 1.0L / sqrtl(x)));
    }
  std::printf("%.4f %.4f\n", e[0], e[1]);
}
"""


def test_within_bounds():
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    emu = os.path.join(ROOT, "tests", "host_emulation")
    h = open(os.path.join(ROOT, "paper_1602_09079_gb300", "csrc", "dg_common.cuh")).read()
    for exact, most in (("return 1.f / x;", 1), ("return 1.f / std::sqrt(x);", 2)):
        assert h.count(exact) == 1
        h = h.replace(exact, f"return moved({exact[7:-1]}, {most});")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "r.cpp"), os.path.join(d, "r")
        open(os.path.join(d, "roots.cuh"), "w").write(h)
        open(src, "w").write(SRC)
        subprocess.run(["g++", "-std=c++20", "-O2", "-pthread", "-I", emu, "-include", os.path.join(emu, "emu.h"), src,
                        "-o", exe], check=True)
        v = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    for x in map(float, v):
        assert x <= 0.52, v
