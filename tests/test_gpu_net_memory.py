"""GPU: device memory of a network that trains."""
import numpy as np
import pytest

import synth
from tests.gpu_common import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


def test_one_pair_needs_no_buffers_beside_the_applications():
    """Training on one pair takes the two fields of an application and one per layer; 16 MB cover the weights, the partial
    sums and the allocator's rounding, a fourth field would not fit into them."""
    dims = (16, 16, 16, 64)
    field = 96 * int(np.prod(dims))
    W = ok.precompute_W(to_dev(synth.random_links(dims, 0.3, 9701)), synth.placeholder_coeffs(0.5), (1, 1, 1, 1), ok.W_F16 | ok.W_LINKS)
    b = to_dev(synth.gaussian_source(dims, 9702).astype(np.complex64))
    x = to_dev(synth.gaussian_source(dims, 9703).astype(np.complex64))
    small = synth.random_links((2, 2, 2, 2), 0.3, 9704)
    Ws = ok.precompute_W(to_dev(small), synth.placeholder_coeffs(0.5), (1, 1, 1, 1), ok.W_F16 | ok.W_LINKS)
    s = to_dev(synth.gaussian_source((2, 2, 2, 2), 9705).astype(np.complex64))
    ok.net_loss_grad(ok.Net(1), Ws, s, 2 * s)   # loads the kernels
    net = ok.Net(1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ok.net_loss_grad(net, W, b, x)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    assert 3 * field <= used < 3 * field + (16 << 20)
