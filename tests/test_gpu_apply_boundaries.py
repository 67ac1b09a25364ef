"""GPU: the FP32 and FP16-W applications in each form of the boundaries (periodic, time antiperiodic, others) and on both sides
of the lookahead's thresholds, against the native FP64 application and the multi-right-hand-side kernel."""
import pytest

import synth
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ok = pytest.importorskip("paper_1311_5029_gb300")


# One multiprocessor's room (1217 sites) and one time slice, where every temporal hop crosses; extents 1 to 3; ragged; time slices
# of W just below and above 5 MiB in FP16 (3386 and 3388 sites) and above 56 MiB in FP32.
@pytest.mark.parametrize("dims", [(11, 11, 11, 1), (1, 3, 2, 300), (13, 7, 5, 9), (16, 16, 16, 4), (2, 1693, 1, 2), (28, 11, 11, 2), (28, 28, 28, 1)])
@pytest.mark.parametrize("bc", [(1, 1, 1, 1), (1, 1, 1, -1), (-1, 1, 1, 1), (1, -1, -1, -1)])
def test_boundary_forms(dims, bc):
    U = synth.device_random_links(dims, 0.3, 8401)
    W = ok.precompute_W(U, synth.random_coeffs(8402), bc, ok.W_F64 | ok.W_F32 | ok.W_F16)
    g = torch.Generator(device="cuda")
    g.manual_seed(8403)
    psi = torch.view_as_complex(torch.randn(synth.lattice_shape(dims) + (4, 3, 2), generator=g, device="cuda", dtype=torch.float64))
    low = psi.to(torch.complex64)
    exp = ok.apply_M(W, psi).cpu().numpy()
    out = torch.full_like(low, float("nan"))
    # the FP32 bar of the parity tests; with the same stored W on both sides it holds for FP16 storage too
    assert rel_l2(ok.apply_M(W, low, out).cpu().numpy(), exp) < 1e-5
    exp16 = ok.apply_M_multi(W, low[None].contiguous(), prec=ok.F32_W16)[0].cpu().numpy()
    out.fill_(float("nan"))
    assert rel_l2(ok.apply_M(W, low, out, prec=ok.F32_W16).cpu().numpy(), exp16) < 1e-5
