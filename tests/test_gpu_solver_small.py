"""GPU: FP32 iterations of small systems (one cluster launch between applications) at the edges of their range."""
import numpy as np
import pytest

import synth
from oracle import wform
from tests.gpu_common import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# 6 V units over 1024-thread blocks, a block per 1536 units and eight at most: one block half empty, one and two
# blocks (256 and 257 sites), all eight; the largest system of the range and the smallest beyond it.
@pytest.mark.parametrize("dims", [(2, 2, 2, 3), (4, 4, 4, 4), (257, 1, 1, 1), (7, 5, 9, 6), (8, 8, 8, 16), (3, 2731, 1, 1)])
@pytest.mark.parametrize("net", [False, True])
def test_small_solves(dims, net):
    bc = (1, 1, 1, -1)
    U = synth.random_links(dims, 0.3, 9501)
    c = synth.placeholder_coeffs(0.6)
    b = synth.gaussian_source(dims, 9502)
    W = ok.precompute_W(to_dev(U), c, bc, ok.W_F32 | ok.W_F64 | (ok.W_LINKS if net else 0))
    A = np.zeros((1, 9, 4, 4), complex)
    A[0, 0] = np.diag([1.0, 0.9, 1.1, 1.0])
    p = ok.Net(1, A) if net else None
    xs = []
    for every in (1, 7):
        if net:
            x, info = ok.bicgstab_net(W, p, to_dev(b), tol=1e-10, check_every=every)
        else:
            x, info = ok.bicgstab(W, to_dev(b), tol=1e-10, mode=ok.SOLVE_MIXED, check_every=every)
        assert info["status"] == 0
        xs.append(x.cpu().numpy())
    assert np.array_equal(xs[0], xs[1])   # the launches are the same, whenever the host looks
    r = np.linalg.norm(b - wform.apply(U, c, xs[0], bc)) / np.linalg.norm(b)
    assert r < 1e-10 and abs(info["true_relres"] - r) < 1e-12


@pytest.mark.parametrize("maxiter", [1, 2, 3])
def test_iteration_limit_in_a_small_system(maxiter):
    dims = (4, 4, 4, 5)
    U = synth.random_links(dims, 0.3, 9511)
    W = ok.precompute_W(to_dev(U), synth.placeholder_coeffs(0.6), (1, 1, 1, 1), ok.W_F32 | ok.W_F64)
    x, info = ok.bicgstab(W, to_dev(synth.gaussian_source(dims, 9512)), tol=1e-14, mode=ok.SOLVE_MIXED, maxiter=maxiter,
                          check_every=1, raise_on_noconv=False)
    assert info["status"] == -4 and info["iters"] == maxiter and torch.isfinite(torch.view_as_real(x)).all()
