"""The kernel for few (patch, object) pairs (a cluster of CTAs per pair,
spread_kernels.cu) against the three-kernel path on the same inputs: the same
arithmetic per line and per frequency, so the objects and dL/da agree bit for
bit (also dL/dO of the object-inferring loss); the loss sums the same FP32 terms
in another partition (1e-6). Frame counts where a CTA takes one or two frames and
where clusters are largest, boxes up to the largest it takes, both layouts."""

import numpy as np
import pytest
import torch

from tests import cases
from tests.test_parity_gpu import _inputs, _plan_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frames,diams,patches,full", [
    (1, (36.0,), 1, False), (2, (4.0, 34.0), 2, False), (8, (32.0,), 1, True), (9, (36.0, 28.0, 20.0), 1, False),
    (12, (36.0,), 1, False), (12, (36.0, 28.0), 14, False), (5, (30.0, 18.0), 25, False),
])
def test_few_pairs_match_three_kernel_path(frames, diams, patches, full):
    wl = [6563.0 * diams[0] / d for d in diams]
    case = cases.make_case(diams=diams, wavelengths=tuple(wl), n_frames=frames, n_modes=9, basis="zernike",
                           n_patches=min(patches, 2), seed=20251000 + frames)
    a32, d32, _ = _inputs(case, full_spectrum=full)
    reps = -(-patches // a32.shape[0])
    a = torch.from_numpy(np.tile(a32, (reps, 1, 1))[:patches]).cuda()
    d = torch.from_numpy(np.tile(d32, (reps, 1, 1, 1, 1))[:patches]).cuda()
    few = _plan_for(case, n_patches=patches, full_spectrum=full)
    split = _plan_for(case, n_patches=patches, full_spectrum=full, split=True)
    assert few.info()["fused_ctas"] > 0
    for _ in range(2):  # the counters are reset between calls
        lf, gf, of = few.loss_grad(a, d, want_object=True)
        ls, gs, os_ = split.loss_grad(a, d, want_object=True)
        assert torch.equal(gf, gs) and torch.equal(of, os_)
        assert ((lf - ls).abs() <= 1e-6 * ls.abs()).all()
    obj = d.mean(2)
    lf, gf, of = few.loss_grad_explicit(a, d, obj)
    ls, gs, os_ = split.loss_grad_explicit(a, d, obj)
    assert torch.equal(gf, gs) and torch.equal(of, os_)
    assert ((lf - ls).abs() <= 1e-6 * ls.abs()).all()
