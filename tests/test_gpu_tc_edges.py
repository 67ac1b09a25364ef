"""GPU: the tensor-core apply and its vector kernels where their tiles, words and divisions end."""
import numpy as np
import pytest

import synth
from oracle import wform
from tests.gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# Right-hand sides below, at and over the 8 of a tile word's first half, and all 16; extents of one, powers of
# two and primes (the divisions of a site's number); fewer sites than warps, and one more than a block's.
# Every product carries an FP16 rounding (2^-11 at most) of an input and of a W entry; over a sum of unrelated
# terms that is 2 * 2^-11 of the output in the 2-norm, and as much again for what cancels.
@pytest.mark.parametrize("dims,bc,nrhs", [((3, 3, 3, 3), (1, 1, 1, 1), 1), ((3, 4, 5, 1), (1, 1, 1, -1), 7), ((8, 4, 3, 16), (1, 1, 1, -1), 8),
                                          ((7, 11, 13, 3), (-1, 1, -1, 1), 9), ((1, 16, 4, 17), (1, 1, 1, 1), 16)])
def test_tensor_core_apply(dims, bc, nrhs):
    U = synth.random_links(dims, 0.3, 9601)
    c = synth.placeholder_coeffs(0.5)
    W = ok.precompute_W(to_dev(U), c, bc, ok.W_F16_TC)
    psi = np.stack([synth.gaussian_source(dims, 9610 + k) for k in range(nrhs)]).astype(np.complex64)
    got = ok.apply_M_multi(W, to_dev(psi), prec=ok.F16_TC).cpu().numpy()
    for k in range(nrhs):
        assert rel_l2(got[k], wform.apply(U, c, psi[k].astype(np.complex128), bc)) < 4 * 2.0 ** -11


@pytest.mark.parametrize("nrhs,mode", [(3, "plain"), (9, "plain"), (9, "defect")])
def test_tensor_core_solves(nrhs, mode):
    dims, bc = (4, 3, 5, 6), (1, 1, 1, -1)
    U = synth.random_links(dims, 0.3, 9651)
    c = synth.placeholder_coeffs(0.8)
    W = ok.precompute_W(to_dev(U), c, bc, ok.W_F16_TC | ok.W_DF64)
    b = np.stack([synth.gaussian_source(dims, 9660 + k) for k in range(nrhs)])
    m = ok.SOLVE_MIXED_TC | (ok.SOLVE_DEFECT if mode == "defect" else 0)
    x, info = ok.bicgstab_multi(W, to_dev(b), tol=1e-10, mode=m)
    x = x.cpu().numpy()
    for k in range(nrhs):
        assert np.linalg.norm(b[k] - wform.apply(U, c, x[k], bc)) < 1e-10 * np.linalg.norm(b[k])
