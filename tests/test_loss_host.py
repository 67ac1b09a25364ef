"""The training loss's sums of squares (csrc/ok_sum3.cuh), compiled for the host, against exact rational sums.

One rounding to FP64 and 2^-68 of it are allowed where the sum runs in floats, and one rounding for each
operation of 8 numbers where it runs in FP64 (below 2^-40 and above 2^40)."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_5029_gb300", "csrc")

HARNESS = r"""
#include "ok_sum3.cuh"
#include <cstdio>
int main(int, char** argv) {
  FILE* f = fopen(argv[1], "rb");
  float2 o[8], x[8];
  while (fread(o, sizeof o, 1, f) == 1 && fread(x, sizeof x, 1, f) == 1) {
    double v[2] = {0.0, 0.0};
    okgb::loss_chunk(o, x, v);
    printf("%a %a\n", v[0], v[1]);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def chunk(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("loss")
    (d / "loss.cu").write_text(HARNESS)
    inc = os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include")
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", inc, "-o", str(d / "loss"), str(d / "loss.cu")], check=True,
                   capture_output=True, timeout=300)

    def run(o, x):
        np.stack([o, x], axis=1).astype(np.float32).tofile(d / "in.bin")
        out = subprocess.run([str(d / "loss"), str(d / "in.bin")], check=True, capture_output=True, text=True).stdout.split()
        return np.array([float.fromhex(t) if "n" not in t else float(t) for t in out]).reshape(-1, 2)

    return run


def _exact(v):
    return sum((Fraction(float(t)) ** 2 for t in v), Fraction(0))


def _check(run, o, x, ulps):
    got = run(o, x)
    for k in range(len(o)):
        n2 = _exact(x[k])
        d2 = sum(((Fraction(float(p)) - Fraction(float(q))) ** 2 for p, q in zip(o[k], x[k])), Fraction(0))
        for g, e in ((got[k, 0], n2), (got[k, 1], d2)):
            assert abs(Fraction(g) - e) <= e * Fraction(ulps, 2 ** 53) + e / 2 ** 68, (k, g, float(e))


def _fields(rng, scale):
    x = (rng.standard_normal((300, 16)) * scale).astype(np.float32)
    return x, (x + (rng.standard_normal((300, 16)) * scale).astype(np.float32)).astype(np.float32)


@pytest.mark.parametrize("k", [-39, -20, 0, 30])
def test_sums_in_floats(chunk, k):
    rng = np.random.default_rng(7)
    x, o = _fields(rng, 2.0 ** k)
    _check(chunk, o, x, 1)


@pytest.mark.parametrize("k", [-60, 50])
def test_sums_in_double(chunk, k):
    rng = np.random.default_rng(8)
    x, o = _fields(rng, 2.0 ** k)
    _check(chunk, o, x, 40)


@pytest.mark.parametrize("k", [-39, -30, 0])
def test_differences_of_a_few_ulps(chunk, k):
    """A well-trained network: P b and x agree to rounding, so the differences' squares are 2^-46 and less of x's."""
    rng = np.random.default_rng(9)
    x, _ = _fields(rng, 2.0 ** k)
    o = x.copy()
    for _ in range(2):
        up = rng.random(o.shape) < 0.5
        o = np.where(up, np.nextafter(o, np.float32(np.inf)), o).astype(np.float32)
    _check(chunk, o, x, 40)


def test_differences_below_the_range_of_floats(chunk):
    """Equal components of order one beside absent ones that differ by far less."""
    rng = np.random.default_rng(10)
    x = rng.standard_normal((50, 16)).astype(np.float32)
    x[:, ::2] = 0
    o = x.copy()
    o[:, ::2] = (1e-25 * rng.standard_normal((50, 8))).astype(np.float32)
    _check(chunk, o, x, 40)


def test_not_finite(chunk):
    x = np.ones((3, 16), np.float32)
    o = np.zeros((3, 16), np.float32)
    o[0, 3], x[1, 4], o[2, 5] = np.nan, np.inf, -np.inf
    got = chunk(o, x)
    assert got[0, 0] == 16 and np.isnan(got[0, 1])
    assert np.isinf(got[1, 0]) and np.isinf(got[1, 1]) and got[2, 0] == 16 and np.isinf(got[2, 1])
