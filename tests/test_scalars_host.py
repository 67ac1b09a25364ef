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
    assert out[:2] == ["0", "0"], out
