"""The entries that the double-float apply walks (csrc/ok_dd_entries.cuh) against the products of csrc/ok_dd_table.cuh: two
lists of the same 148 products in different bases, evaluated on random matrices and spinors."""
import numpy as np
import pytest

from tests.test_dd_entries_host import entries, entries_apply  # noqa: F401 (a fixture)
from tests.test_dd_table_host import Lattice, table, table_apply  # noqa: F401 (a fixture)


@pytest.mark.parametrize("L,bcneg,a,b", [((4, 3, 5, 2), 0b1010, 0.37, -0.61), ((2, 1, 3, 4), 0b0001, 0.61, 0.37), ((3, 3, 3, 3), 0, -0.5, 0.0)])
def test_entries_equal_the_table(entries, table, L, bcneg, a, b):  # noqa: F811
    lat = Lattice(L, bcneg, seed=sum(L) + bcneg)
    err = 0.0
    for s in range(lat.V):
        r = table_apply(lat, s, *table, 0.23, a, b)
        err = max(err, np.abs(r - entries_apply(lat, s, *entries, 0.23, a, b)).max() / np.abs(r).max())
    assert err < 1e-13, err
