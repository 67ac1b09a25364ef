"""Complex division of the solver's scalars (csrc/ok_reduce.cuh), compiled for the host."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_5029_gb300", "csrc")

HARNESS = r"""
#include "ok_reduce.cuh"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
using namespace okgb;
int main() {
  int bad = 0;
  // n / n is 1: |n|^2 / |n|^2 is exact for integers, |n|^2 (1 / |n|^2) is not for every one (7, say)
  for (int n = 1; n <= 2000; ++n) {
    const dcx q = ddiv(dmk(n, 0), dmk(n, 0)), i = ddiv(dmk(0, n), dmk(n, 0));
    if (q.re != 1.0 || q.im != 0.0 || i.re != 0.0 || i.im != 1.0) ++bad;
  }
  printf("%d\n", bad);
  // |b|^2 = 2^-2k, down through the subnormal range: exact powers of two, so the quotient is too
  bad = 0;
  for (int k = 500; k <= 537; ++k) {
    const double s = std::ldexp(1.0, -k);
    const dcx q = ddiv(dmk(3 * s, -s), dmk(s, 0));
    if (q.re != 3.0 || q.im != -1.0) { ++bad; printf("2^-%d: %g %g\n", k, q.re, q.im); }
  }
  printf("%d\n", bad);
  // the shared reciprocal with its correction gives the divisions' own bits, inside and outside its range
  bad = 0;
  std::mt19937_64 g(20131121);
  auto number = [&](int span) {
    unsigned long long u = g();
    u = (u & ~(0x7ffULL << 52)) | ((unsigned long long)(1023 - span / 2 + g() % span) << 52);
    double d;
    std::memcpy(&d, &u, 8);
    return d;
  };
  for (int k = 0; k < 2000000; ++k) {
    const int span = k % 3 == 0 ? 2 : k % 3 == 1 ? 600 : 2040;
    const double x = number(span), y = number(40), d = std::fabs(number(span));
    const dcx q = quot2(x, y, d);
    if (q.re != x / d || q.im != y / d) ++bad;
  }
  for (double d : {5e-324, 1e-310, 0x1p-400, 0x1p400, 0x1.fffffffffffffp400, 1e308})
    for (double x : {0.0, 5e-324, 0x1p-401, 1.0, 0x1p401, 1e308}) {
      const dcx q = quot2(x, -x, d);
      if (q.re != x / d || q.im != -x / d) ++bad;
    }
  printf("%d\n", bad);
  return 0;
}
"""


def test_division_keeps_its_range_and_rounding(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    (tmp_path / "ddiv.cu").write_text(HARNESS)
    inc = os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include")
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", inc, "-o", str(tmp_path / "ddiv"), str(tmp_path / "ddiv.cu")], check=True,
                   capture_output=True, timeout=300)
    out = subprocess.run([str(tmp_path / "ddiv")], check=True, capture_output=True, text=True).stdout.split("\n")
    assert out[:3] == ["0", "0", "0"], out
