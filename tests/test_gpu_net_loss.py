"""GPU: the training loss where P b and x hardly differ."""
import numpy as np
import pytest

import synth
from tests.gpu_common import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# The identity network returns b, so the loss is |b - x|^2 / |x|^2 of the fields as given, up to the roundings of FP64
# sums: a few hundred elements a thread and block trees, far below 1e-12.
@pytest.mark.parametrize("case", ["ulps at 2^-39", "ulps", "tiny beside one"])
def test_loss_of_an_identity_network(case):
    dims = (5, 3, 7, 4)
    W = ok.precompute_W(to_dev(synth.random_links(dims, 0.3, 9601)), synth.placeholder_coeffs(0.5), (1, 1, 1, 1), ok.W_F32 | ok.W_LINKS)
    x = synth.gaussian_source(dims, 9602).astype(np.complex64).view(np.float32).copy()
    rng = np.random.default_rng(3)
    if case == "tiny beside one":
        x[..., ::2] = 0
        b = x.copy()
        b[..., ::2] = 1e-25 * rng.standard_normal(b[..., ::2].shape)
    else:
        if case == "ulps at 2^-39":
            x *= np.float32(2.0 ** -39) / np.abs(x).max()
        b = np.where(rng.random(x.shape) < 0.5, np.nextafter(x, np.float32(np.inf)), x)
    b = b.astype(np.float32)
    d = b.astype(np.float64) - x
    want = np.sum(d * d) / np.sum(x.astype(np.float64) ** 2)
    loss, _ = ok.net_loss_grad(ok.Net(1), W, to_dev(b.view(np.complex64)), to_dev(x.view(np.complex64)))
    assert want > 0 and abs(loss - want) < 1e-12 * want
