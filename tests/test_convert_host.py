"""The integer FP64 -> FP16 conversion of csrc/ok_split.cuh, compiled for the host: bit for bit __double2half."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_5029_gb300", "csrc")

HARNESS = r"""
#include "ok_split.cuh"
#include <cuda_fp16.h>
#include <cmath>
#include <cstdio>
#include <random>
using namespace okgb;
int main() {
  std::mt19937_64 rng(77);
  long long bad = 0;
  auto check = [&](double d) {
    const __half h = __float2half_rn(float_odd_of(d)), k = __double2half(d);
    if (d == d && memcmp(&h, &k, 2) != 0) { if (bad++ < 5) printf("half %a: %a %a\n", d, (double)__half2float(h), (double)__half2float(k)); }
  };
  for (int k = 0; k < 3000000; ++k) {
    const unsigned long long u = rng();
    double d;
    memcpy(&d, &u, 8);
    check(d);
    check(std::ldexp((double)(long long)u, -63 - (int)(rng() % 40)) * 8.0);   // the range of FP16 and below
  }
  for (int e = -160; e <= 140; ++e)      // around powers of two, and halves of an ulp of FP16 and FP32
    for (int t = -300; t <= 300; ++t)
      for (int b : {53, 25, 24, 12, 11}) {
        check(std::ldexp(1.0, e) + t * std::ldexp(1.0, e - b));
        check(-std::ldexp(1.0, e) + std::ldexp(1.0, e - 11) + t * std::ldexp(1.0, e - b - 20));
      }
  const double edge[] = {0.0, -0.0, INFINITY, -INFINITY, NAN, 65504.0, 65519.999999999, 65520.0, 0x1p-24, 0x1p-25, 0x1.0000000000001p-25,
                         0x1p-126, 0x1p-74, 0x1.fffffefffffffp127, 0x1.ffffffp127, 4.9406564584124654e-324};
  for (double d : edge) check(d);
  printf("bad %lld\n", bad);
  return bad != 0;
}
"""


def test_round_to_odd_gives_the_fp16_rounding(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "convert_check.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "convert_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True, timeout=300)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
