"""The FP64 quotient of the barostat's end of a step equals the division's
result, over signs, magnitudes and the values that the step meets."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include "mw_quotient.h"
static uint64_t s = 0x9e3779b97f4a7c15ull;
static uint64_t next() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double unit() { return (double)(next() >> 11) * 0x1p-53; }
static bool same(double x, double y) { return std::memcmp(&x, &y, 8) == 0 || (x != x && y != y); }
int main() {
  long bad = 0;
  auto check = [&](double a, double b) { bad += !same(mw::quotient(a, b), a / b); };
  for (long k = 0; k < 4000000; ++k) {
    const double a = (1.0 + unit()) * (next() & 1 ? 1 : -1), b = (1.0 + unit()) * (next() & 1 ? 1 : -1);
    check(a, b);
    check(std::ldexp(a, (int)(next() % 200) - 100), std::ldexp(b, (int)(next() % 200) - 100));
    check(1.0 + 1e-4 * (a - 1.5), 1.0 + 1e-4 * (b - 1.5));  // edge ratios
  }
  const double inf = std::numeric_limits<double>::infinity(), nan = std::nan("");
  const double v[] = {0.0, -0.0, 1.0, -3.0, 1e-300, 5e-324, 1e300, -1e308, inf, -inf, nan, 1e-35, 1e35, 1e-45, 3e38};
  for (double a : v)
    for (double b : v) check(a, b);
  std::printf("%ld\n", bad);
  return 0;
}
"""


def test_quotient_is_the_division(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "quotient.cc"
    src.write_text(SOURCE)
    exe = tmp_path / "quotient"
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_0809_2811_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0
