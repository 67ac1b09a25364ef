"""GPU: the batched training kernels at the edges of their tiles, groups and value ranges."""
import numpy as np
import pytest

import synth
from oracle import precond
from tests.gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


def _weights(layers, seed):
    w = 0.2 * synth.gaussian(seed, layers * 9 * 16 * 2).reshape(layers, 9, 4, 4, 2)
    w = (w[..., 0] + 1j * w[..., 1]).astype(np.complex64).astype(np.complex128)
    w[:, 0] += np.eye(4)
    return w.astype(np.complex64).astype(np.complex128)


def _fields(dims, n, seed):
    f = np.stack([synth.gaussian_source(dims, seed + k) for k in range(n)]).astype(np.complex64)
    return f, to_dev(f)


# Sites below, at and just over one 32-site tile, and ragged ones over several; batches of one pair, of
# one group and of one pair more than the 64 of a group.
@pytest.mark.parametrize("dims,nb", [((3, 2, 1, 5), 2), ((4, 2, 2, 2), 1), ((3, 11, 1, 1), 3), ((5, 3, 7, 4), 5), ((2, 2, 2, 2), 65)])
def test_training_step_against_the_oracle(dims, nb):
    bc = (1, 1, 1, -1)
    U = synth.random_links(dims, 0.3, 9301)
    W = ok.precompute_W(to_dev(U), synth.placeholder_coeffs(0.5), bc, ok.W_F32 | ok.W_LINKS)
    A = _weights(2, 9302)
    net = ok.Net(2, A)
    (b, bd), (x, xd) = _fields(dims, nb, 9310), _fields(dims, nb, 9810)
    lr = 1e-3
    got = ok.net_train_step(net, W, bd, xd, lr=lr)
    loss, grad = 0.0, np.zeros_like(A)
    for k in range(nb):
        l, g = precond.loss_and_grad(U, A, b[k].astype(np.complex128), x[k].astype(np.complex128), bc)
        loss += l / nb
        grad += g / nb
    assert abs(got - loss) < 1e-5 * loss
    # Adam's first step moves every real parameter by lr g / (|g| + 1e-8).  FP32 fields carry relative
    # errors of some 1e-6 into g, so a component above 1e-3 of the largest moves by lr to 1e-2 of it.
    d = (net.weights - A).view(np.float64)
    g = np.ascontiguousarray(grad).view(np.float64)
    big = np.abs(g) > 1e-3 * np.abs(g).max()
    assert np.abs(d - -lr * g / (np.abs(g) + 1e-8))[big].max() < 1e-2 * lr
    assert np.abs(d).max() < 1.01 * lr


@pytest.mark.parametrize("k", [-45, 45])
def test_loss_and_gradient_do_not_depend_on_the_fields_scale(k):
    """Fields times 2^k: the loss's squares leave the range of its FP32 sums and are taken in FP64."""
    dims, bc = (5, 3, 7, 4), (1, 1, 1, 1)
    U = synth.random_links(dims, 0.3, 9401)
    W = ok.precompute_W(to_dev(U), synth.placeholder_coeffs(0.5), bc, ok.W_F32 | ok.W_LINKS)
    net = ok.Net(2, _weights(2, 9402))
    (_, b), (_, x) = _fields(dims, 1, 9410), _fields(dims, 1, 9420)
    l0, g0 = ok.net_loss_grad(net, W, b[0], x[0])
    l1, g1 = ok.net_loss_grad(net, W, b[0] * 2.0 ** k, x[0] * 2.0 ** k)
    assert abs(l1 - l0) < 1e-10 * l0     # powers of two are exact; the double-float sums carry 2^-44
    # the gradient is linear in both fields and carries 1 / |x|^2, whose FP32 rounding may differ
    assert rel_l2(g1, g0) < 1e-6
