"""Data spectra beside the element at 0, against the definition in 64 bits: the
patch's mean is far larger than its deviations, and their spectrum has to be as
accurate as FP32 transforms of the deviations alone make it. Two line
transforms of 9e-8 each, the subtraction and two window products of 3.4e-8 each
and the mean's own rounding add up to 1.6e-7 norm-wise; the bound is 4e-7 (with
the mean in the pixels that are transformed it was 1.5e-6 to 2e-6)."""

import numpy as np
import pytest
import torch

from oracle import patches as opatches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,overlap", [(48, 24), (48, 19), (64, 32), (64, 29), (96, 48), (96, 53), (128, 64), (128, 67)])
def test_spectra_of_the_deviations(n, overlap):
    from paper_2505_10639_gb300.mfbd import Plan
    h = 2 * (n - overlap) + n
    frames = (1.0 + 0.1 * np.random.default_rng(n + overlap).standard_normal((1, 5, h, h))).astype(np.float32)
    plan = Plan(n, 9, [0.5 * n], [6563.0], 5, 8, gamma=1e-3)
    d = plan.spectra_from_frames(torch.from_numpy(frames).cuda(), overlap, n // 8).cpu().numpy()
    ref = np.asarray(opatches.spectra_from_frames(frames.astype(np.float64), n, overlap, n // 8))[..., :n // 2 + 1]
    assert np.abs(d[..., 0, 0] - ref[..., 0, 0]).max() <= 3 * 2.0 ** -24 * np.abs(ref[..., 0, 0]).max()
    d[..., 0, 0] = ref[..., 0, 0] = 0
    err = np.linalg.norm(d - ref) / np.linalg.norm(ref)
    assert err <= 4e-7, err
