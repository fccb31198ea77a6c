"""The object-inferring loss on the general-size kernels at the frame counts
where their reduction changes its form (8 and 16 frames held in registers, more
read in chunks) and for the 64 px plans of more than 12 frames, against the FP64
oracle: loss, dL/da and dL/dconj(O), in both spectrum layouts. Tolerances are
those of the smaller frame counts (1e-5 relative, 1e-4 and OBJ_GRAD_RTOL
norm-wise)."""

import numpy as np
import pytest
import torch

from oracle import mfbd as omfbd
from tests import cases
from tests.test_explicit_gpu import OBJ_GRAD_RTOL, _given_objects, _plan
from tests.test_parity_gpu import _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("n_pix,diams,frames", [
    (64, (36.0,), 13), (64, (36.0, 28.0), 16), (64, (36.0,), 17), (64, (30.0,), 33),
    (48, (22.0,), 8), (96, (40.0,), 9), (48, (26.0,), 16), (96, (40.0,), 17),
])
def test_explicit_loss_by_frame_count(n_pix, diams, frames, full):
    case = cases.make_case(n_pix=n_pix, diams=diams, wavelengths=(6563.0, 8542.0)[:len(diams)], n_frames=frames,
                           n_modes=8, basis="zernike", n_patches=2, seed=20251400 + frames)
    a32, d32, d_or = _inputs(case, full_spectrum=full)
    if full:  # the kernels read the columns kx <= N/2 of full spectra
        d_or = omfbd.full_from_half(omfbd.half_spectrum(d_or), n_pix)
    a64 = a32.astype(np.float64)
    o_gpu, o_full = _given_objects(case, d_or, a64, frames, full)
    loss, grad, gobj = _plan(case, full_spectrum=full).loss_grad_explicit(
        torch.from_numpy(a32).cuda(), torch.from_numpy(d32).cuda(), torch.from_numpy(np.ascontiguousarray(o_gpu)).cuda())
    loss, grad, gobj = loss.cpu().numpy(), grad.cpu().numpy(), gobj.cpu().numpy().astype(np.complex128)
    for p in range(a32.shape[0]):
        lo, go, gob = omfbd.explicit_loss_grad_patch(case["setup"], a64[p], d_or[p], o_full[p])
        want = gob if full else omfbd.half_spectrum(gob)
        assert abs(loss[p] - lo) <= 1e-5 * abs(lo)
        assert np.linalg.norm(grad[p] - go) <= 1e-4 * np.linalg.norm(go)
        assert np.linalg.norm(gobj[p] - want) <= OBJ_GRAD_RTOL * np.linalg.norm(want)
