"""GPU: the FP32 application against the native FP64 one, and the FP16-W application against the
multi-right-hand-side kernel on the same FP16 W (both pinned to the oracle by the parity tests), at the
sizes where their kernels and tile assignments change."""
import numpy as np
import pytest

import synth
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# One site; a block of 16 sites and one more; the last lattice of the small kernel on 152 multiprocessors
# (1216 sites) and the next; ragged tiles; whole rounds of tiles and a spread last round (4224 tiles);
# time slices of W above the thresholds of the lookahead (28^3: FP32; 17 x 17 x 17: FP16).
@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (2, 2, 2, 2), (17, 1, 1, 1), (8, 8, 19, 1), (1217, 1, 1, 1), (5, 7, 11, 5), (3, 2, 401, 1),
                                  (16, 16, 16, 33), (28, 28, 28, 2), (17, 17, 17, 3)])
@pytest.mark.parametrize("bct", [1, -1])
def test_low_precision_applies_against_fp64(dims, bct):
    bc = (bct, 1, 1, bct)
    U = synth.device_random_links(dims, 0.3, 8201)
    W = ok.precompute_W(U, synth.random_coeffs(8202), bc, ok.W_F64 | ok.W_F32 | ok.W_F16)
    g = torch.Generator(device="cuda")
    g.manual_seed(8203)
    psi = torch.view_as_complex(torch.randn(synth.lattice_shape(dims) + (4, 3, 2), generator=g, device="cuda", dtype=torch.float64))
    exp = ok.apply_M(W, psi).cpu().numpy()
    out = torch.full_like(psi, float("nan")).to(torch.complex64)
    low = psi.to(torch.complex64)
    # the FP32 bar of the parity tests; with the same stored W on both sides it holds for FP16 storage too
    assert rel_l2(ok.apply_M(W, low, out).cpu().numpy(), exp) < 1e-5
    exp16 = ok.apply_M_multi(W, low[None].contiguous(), prec=ok.F32_W16)[0].cpu().numpy()
    out.fill_(float("nan"))
    assert rel_l2(ok.apply_M(W, low, out, prec=ok.F32_W16).cpu().numpy(), exp16) < 1e-5


@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (31, 1, 1, 1), (3, 11, 1, 1), (5, 7, 11, 5)])
def test_double_float_apply_against_fp64(dims):
    """Tiles of 32 sites: one site, one short of a tile, one over, ragged."""
    bc = (1, -1, 1, -1)
    U = synth.device_random_links(dims, 0.3, 8301)
    c = synth.random_coeffs(8302)
    W, D = ok.precompute_W(U, c, bc, ok.W_F64), ok.precompute_W(U, c, bc, ok.W_DF64)
    g = torch.Generator(device="cuda")
    g.manual_seed(8303)
    psi = torch.view_as_complex(torch.randn(synth.lattice_shape(dims) + (4, 3, 2), generator=g, device="cuda", dtype=torch.float64))
    exp, got = ok.apply_M(W, psi), ok.apply_M(D, psi)
    assert rel_l2(got.cpu().numpy(), exp.cpu().numpy()) < 1e-12
    assert abs(ok.true_residual(D, exp * 0.5, psi) - 1.0) < 1e-10     # |exp / 2 - M psi| / |exp / 2| = 1
