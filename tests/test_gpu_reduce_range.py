"""GPU: inner products of FP32 applications of fields whose totals exceed FP32's range."""
import numpy as np
import pytest

import synth
from tests.gpu_common import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# Fields of 2^56: a component's square is some 2^116, the sum over the 230400 components beyond 2^128.  The bar is that of FP32
# products summed in FP32 over a few elements.
@pytest.mark.parametrize("prec", ["f32", "f32_w16"])
@pytest.mark.parametrize("k", [0, 56])
def test_sums_beyond_the_range_of_fp32(prec, k):
    dims = (12, 10, 8, 10)
    W = ok.precompute_W(to_dev(synth.random_links(dims, 0.3, 4701)), synth.placeholder_coeffs(0.5), (1, 1, 1, -1), ok.W_F32 | ok.W_F16)
    p = ok.F32 if prec == "f32" else ok.F32_W16
    psi = to_dev((synth.gaussian_source(dims, 4702) * 2.0 ** k).astype(np.complex64))
    y = to_dev((synth.gaussian_source(dims, 4703) * 2.0 ** k).astype(np.complex64))
    out, (dot, _) = ok.apply_M_reduce(W, psi, y, ok.REDUCE_DOT, prec=p)
    o, s = out.cpu().numpy().astype(np.complex128), y.cpu().numpy().astype(np.complex128)
    scale = np.linalg.norm(o) * np.linalg.norm(s)
    assert abs(dot - np.vdot(s, o)) < 1e-6 * scale
    out, (ts, tt) = ok.apply_M_reduce(W, psi, y, ok.REDUCE_TS, prec=p)
    assert abs(ts - np.vdot(o, s)) < 1e-6 * scale and abs(tt - np.vdot(o, o).real) < 1e-6 * np.vdot(o, o).real
