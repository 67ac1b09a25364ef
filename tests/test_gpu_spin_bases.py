"""GPU: the applications for every balance of the two-hop scalars a = c4 / (2 u0) and
b = (c1 + 2 c2) / (4 u0), which the kernels fold into the spinors in ways that depend on the larger."""
import numpy as np
import pytest

import synth
from oracle import wform
from tests.gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# a > b, a < b, a = 0, b = 0, b < 0 and both zero.
@pytest.mark.parametrize("c1,c2,c4", [(0.01, 0.01, 0.3), (0.5, 0.3, 0.02), (0.05, 0.02, 0.0), (0.0, 0.0, 0.03), (-0.4, 0.1, 0.02), (0.0, 0.0, 0.0)])
def test_two_hop_scalars(c1, c2, c4):
    dims, bc = (5, 4, 3, 7), (1, -1, 1, -1)
    U = synth.random_links(dims, 0.4, 8101)
    c = synth.random_coeffs(8102).replace(c1=c1, c2=c2, c4=c4)
    psi = synth.gaussian_source(dims, 8103)
    exp = wform.apply(U, c, psi, bc)
    # the bars of the parity tests: 1e-12 in FP64 and double-float, 1e-5 in FP32
    for precs, prec, dtype, tol in ((ok.W_F64, ok.F64, np.complex128, 1e-12), (ok.W_DF64, ok.F64, np.complex128, 1e-12),
                                    (ok.W_F32, ok.F32, np.complex64, 1e-5)):
        W = ok.precompute_W(to_dev(U), c, bc, precs)
        got = ok.apply_M(W, to_dev(psi.astype(dtype)), prec=prec).cpu().numpy()
        assert rel_l2(got, exp) < tol
