"""GPU: the gradient's sums, where every rounding shows and where FP32 cannot hold them."""
import numpy as np
import pytest

import synth
from oracle import precond
from tests.gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# Integer fields on unit links under the identity network: a site's six products of parts up to 1448 stay below 2^24 and are
# exact in FP32, the sums over sites are not.  |x|^2 = 2^20, so g = (b - x) / |x|^2 is exact as well, and the gradient is
# an integer multiple of 2^-19 that the FP64 sums hold exactly.
@pytest.mark.parametrize("dims", [(24, 24, 24, 4), (5, 3, 7, 4), (38, 32, 8, 8)])
def test_sums_of_integers_are_exact(dims):
    X, Y, Z, T = dims
    U = np.zeros((T, Z, Y, X, 4, 3, 3), complex)
    U[...] = np.eye(3)
    W = ok.precompute_W(to_dev(U), synth.placeholder_coeffs(0.5), (1, 1, 1, 1), ok.W_F16 | ok.W_LINKS)
    rng = np.random.default_rng(11)
    re, im = rng.integers(-1448, 1449, size=(2, T, Z, Y, X, 4, 3))
    re[0, 0, 0, 0] = im[0, 0, 0, 0] = 0
    gr, gi = re.copy(), im.copy()   # (b - x), in integers
    gr[0, 0, 0, 0, 0, 0] = -1024
    x = np.zeros((T, Z, Y, X, 4, 3), np.complex64)
    x[0, 0, 0, 0, 0, 0] = 1024.0
    loss, grad = ok.net_loss_grad(ok.Net(1), W, to_dev((re + 1j * im).astype(np.complex64)), to_dev(x))
    axes = {0: 3, 1: 2, 2: 1, 3: 0}
    for d in range(9):
        wr, wi = re, im
        if d:
            mu, step = (d - 1) // 2, 1 if d % 2 else -1
            wr, wi = np.roll(re, -step, axes[mu]), np.roll(im, -step, axes[mu])
        a, b = gr.reshape(-1, 4, 3), gi.reshape(-1, 4, 3)
        p, q = wr.reshape(-1, 4, 3), wi.reshape(-1, 4, 3)
        want_re = np.einsum("xsc,xtc->st", a, p) + np.einsum("xsc,xtc->st", b, q)   # g conj(w)
        want_im = np.einsum("xsc,xtc->st", b, p) - np.einsum("xsc,xtc->st", a, q)
        assert np.array_equal(grad[0, d].real * 2.0 ** 19, want_re) and np.array_equal(grad[0, d].imag * 2.0 ** 19, want_im), d
    assert loss == (np.sum(gr * gr) + np.sum(gi * gi)) / 2.0 ** 20


@pytest.mark.parametrize("k", [57, 60])
def test_products_beyond_the_range_of_the_float_sums(k):
    """b of 2^k against x of order one: the products reach 2^100 and more, and their sums are taken in FP64."""
    dims, bc = (5, 3, 7, 4), (1, 1, 1, -1)
    U = synth.random_links(dims, 0.3, 9801)
    W = ok.precompute_W(to_dev(U), synth.placeholder_coeffs(0.5), bc, ok.W_F16 | ok.W_LINKS)
    A = (0.1 * synth.gaussian(9802, 2 * 9 * 16 * 2).reshape(2, 9, 4, 4, 2)).view(np.complex128)[..., 0]
    A[:, 0] += np.eye(4)
    A = A.astype(np.complex64).astype(np.complex128)
    b = (synth.gaussian_source(dims, 9803) * 2.0 ** k).astype(np.complex64)
    x = synth.gaussian_source(dims, 9804).astype(np.complex64)
    loss, grad = ok.net_loss_grad(ok.Net(2, A), W, to_dev(b), to_dev(x))
    l, g = precond.loss_and_grad(U, A, b.astype(np.complex128), x.astype(np.complex128), bc)
    assert np.isfinite(grad).all() and abs(loss - l) < 1e-5 * l and rel_l2(grad, g) < 1e-5
