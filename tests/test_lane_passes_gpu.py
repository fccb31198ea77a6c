"""The CTA-per-unit passes (lines of eight lanes) at the edges of their
buffers, against the FP64 oracle: pupil boxes of a few pixels, of exactly half
the patch (the last box of the half-box buffer), just beyond it and of the
whole patch (the full-box buffer), with and without the recomputed field, for
every patch size. Tolerances are those of the FP32 path (loss 1e-5 relative,
dL/da and object 1e-4 norm-wise)."""

import pytest

from tests import cases
from tests.test_parity_gpu import _check, _inputs, _oracle, _plan_for, _run_fused

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recompute", [False, True])
@pytest.mark.parametrize("n_pix,diams", [
    (48, (24.0, 6.0)), (48, (26.0,)), (48, (48.0, 20.0)),
    (64, (32.0, 8.0)), (64, (34.0,)), (64, (64.0,)),
    (96, (48.0, 10.0)), (96, (50.0,)), (96, (96.0, 40.0)),
    (128, (64.0, 12.0)), (128, (66.0,)), (128, (128.0,)),
])
def test_pupil_box_edges(n_pix, diams, recompute):
    case = cases.make_case(n_pix=n_pix, diams=diams, wavelengths=(6563.0, 8542.0)[:len(diams)], n_frames=3,
                           n_modes=6, basis="zernike", n_patches=2, seed=20250600 + n_pix)
    a32, d32, d_or = _inputs(case)
    plan = _plan_for(case, recompute=recompute, generic=True)
    assert plan.info()["slots_per_cta"] == 0  # the general-size kernels
    loss, grad, obj = _run_fused(plan, a32, d32)
    _check(case, loss, grad, obj, _oracle(case, a32, d_or))
