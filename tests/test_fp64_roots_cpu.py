"""The FP64 path's own reciprocal, reciprocal square root, square root and
two-thirds power (dg_common.cuh), compiled for the host, against long double
over the exponent range: significands at the ends and in between, exact powers,
arguments that take the library function. Bounds: 0.52 units in the last place
for the reciprocals (60 bits before the rounding), 1.6 for the square root (two
roundings), 3 for the power (4 roundings of at most half a unit each, amplified
by at most 1.5)."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "dg_common.cuh"
#include <random>
using namespace dg;
static double ulps(double y, long double t) {
  const double a = std::fabs((double)t);
  return (double)(fabsl((long double)y - t) / (long double)(std::nextafter(a, INFINITY) - a));
}
int main() {
  std::mt19937_64 g(1);
  double e[4] = {0, 0, 0, 0};
  for (long i = 0; i < 2000000; ++i) {
    unsigned long long b = g();
    int ex = i % 3 ? 100 + (int)((b >> 52) % 1800) : 1020 + (int)(i % 7);
    b = (b & 0xfffffffffffffull) | ((unsigned long long)ex << 52);
    if (i % 5 == 0) b &= ~0xffffffffffull;
    if (i % 7 == 0) b |= 0xffffffffffff0ull;
    double x;
    std::memcpy(&x, &b, 8);
    if (rcp64(-x) != -rcp64(x)) return 1;
    e[0] = std::max(e[0], ulps(rcp64(x), 1.0L / x));
    e[1] = std::max(e[1], ulps(rsqrt64(x), 1.0L / sqrtl(x)));
    e[2] = std::max(e[2], ulps(sqrt64(x), sqrtl(x)));
    e[3] = std::max(e[3], ulps(pow_2_3(x), powl(cbrtl(x), 2)));
  }
  const bool special = std::isinf(rcp64(0.0)) && rcp64(INFINITY) == 0.0 && std::isinf(rsqrt64(0.0)) &&
                       std::isnan(rsqrt64(-1.0)) && sqrt64(-1.0) == 0.0 && sqrt64(0.0) == 0.0 && pow_2_3(0.0) == 0.0 &&
                       std::isnan(rcp64(NAN)) && std::isnan(rsqrt64(NAN)) && rcp64(1e-310) == 1.0 / 1e-310 &&
                       rcp64(1.0) == 1.0 && rsqrt64(4.0) == 0.5 && sqrt64(9.0) == 3.0 && pow_2_3(-8.0) == 4.0;
  std::printf("%d %.4f %.4f %.4f %.4f\n", special, e[0], e[1], e[2], e[3]);
}
"""


def test_within_bounds():
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    emu = os.path.join(ROOT, "tests", "host_emulation")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "r.cpp"), os.path.join(d, "r")
        open(src, "w").write(SRC)
        subprocess.run(["g++", "-std=c++20", "-O2", "-pthread", "-I", emu, "-include", os.path.join(emu, "emu.h"), "-I",
                        os.path.join(ROOT, "paper_1602_09079_gb300", "csrc"), src, "-o", exe], check=True)
        v = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert v[0] == "1"
    for x, bound in zip(map(float, v[1:]), (0.52, 0.52, 1.6, 3.0)):
        assert x <= bound, v
