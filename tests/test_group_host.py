"""The size of a training group when memory is short (csrc/ok_group.cuh), with a fake of the allocation."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1311_5029_gb300", "csrc")

# Arguments: the largest group that memory holds, then the groups wanted by one step after another.  Prints for each step
# the group it runs with and the sizes it asked memory for.
HARNESS = r"""
#include "ok_group.cuh"
#include <cstdio>
#include <cstdlib>
int main(int argc, char** argv) {
  const int room = atoi(argv[1]);
  int have = 0, most = 0;
  for (int k = 2; k < argc; ++k) {
    printf("step");
    const int g = okgb::grow_group(atoi(argv[k]), have, most, [&](int q) { printf(" %d", q); return q <= room; });
    printf(" -> %d\n", g);
    have = g;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("group")
    (d / "group.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(d / "group"), str(d / "group.cu")], check=True, capture_output=True,
                   timeout=300)

    def run(*args):
        out = subprocess.run([str(d / "group")] + [str(a) for a in args], check=True, capture_output=True, text=True).stdout
        return [line.replace("step", "").split() for line in out.splitlines()]

    return run


def test_a_group_that_fits_is_asked_for_once(steps):
    assert steps(64, 5, 5, 3, 17, 17) == [["5", "->", "5"], ["->", "5"], ["->", "5"], ["17", "->", "17"], ["->", "17"]]


def test_a_refused_group_is_halved_and_not_asked_for_again(steps):
    assert steps(10, 64, 64, 64) == [["64", "32", "16", "8", "->", "8"], ["->", "8"], ["->", "8"]]


def test_a_group_in_use_stays_when_a_larger_one_is_refused(steps):
    assert steps(4, 4, 64, 64, 5) == [["4", "->", "4"], ["64", "32", "16", "8", "->", "4"], ["->", "4"], ["->", "4"]]


def test_nothing_fits(steps):
    assert steps(0, 3, 3) == [["3", "1", "->", "0"], ["3", "1", "->", "0"]]
