"""The entries that the double-float apply walks (csrc/ok_dd_entries.cuh), built on the host and
evaluated on random matrices and spinors against the products of the table in ok_dd_table.cuh, whose own
test compares them with a transcription of the templated apply."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from tests.test_dd_table_host import CSRC, Lattice, mdv, mv, templated_apply

HARNESS = r"""
#include "ok_dd_entries.cuh"
#include <cstdio>
using namespace okgb::ddent;
int main() {
  const Table t = build();
  for (int h = 0; h < HOPS; ++h) printf("H %d %d %d %d\n", t.d[h][0], t.d[h][1], t.d[h][2], t.d[h][3]);
  for (int w = 0; w < 4; ++w)
    for (int i = 0; i < N_ALL; ++i) printf("E %d %d %d %d\n", t.e[w][i].m, t.e[w][i].hop, t.e[w][i].flags, t.e[w][i].src);
  printf("N %d %d %d %d\n", N_TWO, N_D, N_S, N_ALL);
  return 0;
}
"""


@pytest.fixture(scope="module")
def entries(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("ddent")
    (d / "dump.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-o", str(d / "dump"), str(d / "dump.cu")], check=True, capture_output=True,
                   timeout=300)
    rows = [line.split() for line in subprocess.run([str(d / "dump")], check=True, capture_output=True, text=True).stdout.splitlines()]
    hops = [list(map(int, r[1:])) for r in rows if r[0] == "H"]
    ents = [list(map(int, r[1:])) for r in rows if r[0] == "E"]
    ends = [list(map(int, r[1:])) for r in rows if r[0] == "N"][0]
    assert len(hops) == 27 and len(ents) == 148
    return hops, [ents[37 * w:37 * w + 37] for w in range(4)], ends


def entries_apply(lat, s, hops, ents, ends, c0q, a, b):
    """M psi at site s as the kernel's four warps compute it."""
    c = lat.coords(s)
    big, r, a_big = (a, b / a, True) if abs(a) >= abs(b) else (b, a / b, False)
    D, S, O = [], [], []
    for w in range(4):
        acc = np.zeros(3, complex)
        for i, (m, h, flags, src) in enumerate(ents[w]):
            n, neg = lat.nbr(c, hops[h])
            x = lat.psi[n].reshape(4, 3)
            v, unit = x[src & 3], src >> 4
            if unit:
                y = 1j ** (unit - 1) * x[src >> 2 & 3]
                if i < ends[0]:
                    v, y = (v, r * y) if a_big else (r * v, y)
                v = v + y
            if neg != bool(flags & 2):
                v = -v
            acc = acc + (mdv(lat.W[n][m], v) if flags & 1 else mv(lat.W[s][m], v))
            if i == ends[0] - 1:
                acc = acc * big
            elif i + 1 in ends[1:]:
                (D if i + 1 == ends[1] else S if i + 1 == ends[2] else O).append(acc)
                acc = np.zeros(3, complex)
    x = lat.psi[s].reshape(4, 3)
    out = []
    for w in range(4):
        h, q = divmod(w, 2)
        o = O[q] + O[2 + q] if h == 0 else 1j * (O[q] - O[2 + q])
        out.append(S[q] + (1 - 2 * h) * S[2 + q] + 2 * (D[w] + o) + 4 * c0q * x[w])
    return np.concatenate(out)


@pytest.mark.parametrize("L,bcneg,a,b", [((4, 3, 5, 2), 0b1010, 0.37, -0.61), ((2, 1, 3, 4), 0b0001, 0.61, 0.37), ((3, 3, 3, 3), 0, -0.5, 0.0)])
def test_entries_equal_templated_apply(entries, L, bcneg, a, b):
    hops, ents, ends = entries
    lat = Lattice(L, bcneg, seed=sum(L) + bcneg)
    err = 0.0
    for s in range(lat.V):
        r = templated_apply(lat, s, 0.23, a, b)
        err = max(err, np.abs(r - entries_apply(lat, s, hops, ents, ends, 0.23, a, b)).max() / np.abs(r).max())
    assert err < 1e-13, err
