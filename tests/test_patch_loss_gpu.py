"""A patch's loss and object do not depend on how many patches its plan holds:
at 64 px and up to 12 frames, plans of few (patch, object) pairs run a cluster of
CTAs per pair, the others one CTA per pair, and both give the same bits (also
with the objects given)."""

import numpy as np
import pytest
import torch

from tests import cases
from tests.test_parity_gpu import _inputs, _plan_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frames,diams,full", [
    (1, (36.0,), False), (2, (30.0,), True), (4, (28.0, 20.0), False), (7, (36.0, 28.0, 20.0), False), (8, (32.0,), False),
    (9, (34.0,), False), (11, (36.0, 24.0), True), (12, (36.0, 28.0), False),
])
def test_patch_loss_and_object_by_plan_size(frames, diams, full):
    wl = [6563.0 * diams[0] / d for d in diams]
    case = cases.make_case(diams=diams, wavelengths=tuple(wl), n_frames=frames, n_modes=9, basis="zernike",
                           n_patches=3, seed=20251200 + frames)
    a32, d32, _ = _inputs(case, full_spectrum=full)
    tile = 110  # 330 patches: more pairs than clusters of one CTA fit the GPU
    a, d = torch.from_numpy(a32).cuda(), torch.from_numpy(d32).cuda()
    many_a, many_d = a.repeat(tile, 1, 1), d.repeat(tile, 1, 1, 1, 1)
    few, many = (_plan_for(case, n_patches=n, full_spectrum=full) for n in (3, 3 * tile))
    lf, _, of = few.loss_grad(a, d, want_object=True)
    lm, _, om = many.loss_grad(many_a, many_d, want_object=True)
    assert torch.equal(lm, lf.repeat(tile)) and torch.equal(om, of.repeat(tile, 1, 1, 1))
    obj = d.mean(2).contiguous()
    lf, _, of = few.loss_grad_explicit(a, d, obj)
    lm, _, om = many.loss_grad_explicit(many_a, many_d, obj.repeat(tile, 1, 1, 1))
    assert torch.equal(lm, lf.repeat(tile)) and torch.equal(om, of.repeat(tile, 1, 1, 1))
    few.check()
    many.check()
    assert np.isfinite(lf.cpu().numpy()).all()


@pytest.mark.parametrize("frames,diam,sizes", [
    (1, 36.0, (60, 142, 200)), (4, 28.0, (30, 70)), (10, 36.0, (11, 28)), (12, 28.0, (9, 22, 45)),
])
def test_patch_results_across_the_cluster_rule(frames, diam, sizes):
    """Plan sizes well below and near the most clusters that fit the GPU at once (where the launch is not chained, or
    a CTA takes two frames): the bits of a single patch's plan, call after call."""
    case = cases.make_case(diams=(diam,), wavelengths=(6563.0,), n_frames=frames, n_modes=9, basis="zernike",
                           n_patches=1, seed=20251300 + frames)
    a32, d32, _ = _inputs(case)
    a, d = torch.from_numpy(a32).cuda(), torch.from_numpy(d32).cuda()
    one = _plan_for(case, n_patches=1)
    l1, _, o1 = one.loss_grad(a, d, want_object=True)
    for n in sizes:
        plan = _plan_for(case, n_patches=n)
        an, dn = a.repeat(n, 1, 1), d.repeat(n, 1, 1, 1, 1)
        out = [plan.loss_grad(an, dn, want_object=True) for _ in range(6)]
        plan.check()
        for ln, gn, on in out:
            assert torch.equal(ln, l1.repeat(n)) and torch.equal(on, o1.repeat(n, 1, 1, 1)), n
            assert torch.equal(gn, gn[:1].repeat(n, 1, 1)), n
