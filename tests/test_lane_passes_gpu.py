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


@pytest.mark.parametrize("shapes", [
    [(48, 24.0, 3)],                                                     # one small size: the smallest buffer
    [(48, 26.0, 1), (64, 64.0, 2), (96, 50.0, 3), (128, 66.0, 2)],       # boxes wider than half: the full-box buffer
    [(48, 20.0, 2), (64, 32.0, 5), (96, 48.0, 1), (128, 64.0, 3)],       # odd unit counts, boxes of exactly half
])
def test_batch_box_and_unit_edges(shapes):
    """Uneven batches whose units do not fill their items, against plans of the single problems."""
    import torch

    from paper_2505_10639_gb300.mfbd import Batch, Problem
    data = []
    for i, (n, diam, frames) in enumerate(shapes):
        case = cases.make_case(n_pix=n, diams=(diam,), wavelengths=(6563.0,), n_frames=frames, n_modes=6,
                               basis="zernike", n_patches=1, seed=20250700 + i)
        a32, d32, d_or = _inputs(case)
        data.append((case, a32, d32, _oracle(case, a32, d_or)))
    b = Batch([Problem(c["n_pix"], 1, c["diams"], c["wavelengths"], c["n_frames"], c["n_modes"],
                       gamma=c["setup"].gamma) for c, _, _, _ in data])
    coeffs = Batch.pack([torch.from_numpy(a).cuda() for _, a, _, _ in data])
    spectra = Batch.pack([torch.from_numpy(d).cuda() for _, _, d, _ in data])
    for variant in (0, 1):
        b.set_schedule("one_launch", 0, 0, variant)
        out = b.loss_grad(coeffs, spectra, want_object=True)
        b.check()
        loss, grad, obj = (b.unpack(t, k) for t, k in zip(out, ("loss", "grad", "object")))
        for i, (case, _, _, ref) in enumerate(data):
            _check(case, loss[i].cpu().numpy(), grad[i].cpu().numpy(), obj[i].cpu().numpy().astype("complex128"), ref)


@pytest.mark.parametrize("frames", [1, 8, 9, 16, 17, 32, 33, 64, 65, 129])
@pytest.mark.parametrize("n_pix,diams", [(48, (20.0, 24.0)), (96, (40.0,))])
def test_frame_reduction_frame_counts(n_pix, diams, frames):
    """The frame reduction where its register forms (8, 16, 32 frames) end and its chunked form begins."""
    case = cases.make_case(n_pix=n_pix, diams=diams, wavelengths=(6563.0, 8542.0)[:len(diams)], n_frames=frames,
                           n_modes=5, basis="zernike", n_patches=1, seed=20250800 + frames)
    a32, d32, d_or = _inputs(case)
    loss, grad, obj = _run_fused(_plan_for(case), a32, d32)
    _check(case, loss, grad, obj, _oracle(case, a32, d_or))


@pytest.mark.parametrize("atoms", [1, 2, 3])
def test_dictionary_units_beyond_one_wave(atoms):
    """More units than resident CTAs (a CTA takes several, its exchange buffers alternating across them): copies of a
    patch get the bits of the first."""
    import numpy as np

    from paper_2505_10639_gb300 import synth
    from tests.test_dict_gpu import _check as check_dict
    from tests.test_dict_gpu import _oracle as oracle_dict
    from tests.test_dict_gpu import _run as run_dict
    case = list(synth.dictionary_case(20250900 + atoms, 2, 2, 3, atoms))
    one = run_dict(tuple(case))
    many = list(case)
    for i in (3, 4, 5):
        many[i] = np.tile(case[i], (60,) + (1,) * (case[i].ndim - 1))
    loss, go, ga = run_dict(tuple(many))
    for r in range(60):
        assert np.array_equal(loss[2 * r:2 * r + 2], one[0])
        assert np.array_equal(go[2 * r:2 * r + 2], one[1]) and np.array_equal(ga[2 * r:2 * r + 2], one[2])
    check_dict(0, *one, oracle_dict(tuple(case), 0))


@pytest.mark.parametrize("n,h,w,overlap,border,frames", [
    (48, 131, 140, 17, 9, 90),    # more units than one wave of the persistent grid at every size, strides and
    (64, 167, 201, 29, 13, 60),   # widths that are no multiples of four, and a remainder
    (96, 203, 299, 53, 1, 40),
    (128, 261, 325, 67, 24, 20),
])
def test_spectra_beyond_one_wave(n, h, w, overlap, border, frames):
    """Data spectra of any size and alignment; 1e-5 relative (max-norm), as for the other spectra."""
    import numpy as np
    import torch

    from oracle import mfbd as omfbd
    from oracle import patches as opatches
    from paper_2505_10639_gb300.mfbd import Plan
    g = np.random.default_rng(n)
    data = (1.0 + 0.1 * g.standard_normal((2, frames, h, w))).astype(np.float32)
    grid = opatches.patch_grid(h, w, n, overlap)
    plan = Plan(n, len(grid), [0.4 * n, 0.3 * n], [6563.0, 6563.0 * 4 / 3], frames, 8, gamma=1e-3)
    units = len(grid) * 2 * frames
    assert units > 152 * (2 if n == 128 else 4)
    d = plan.spectra_from_frames(torch.from_numpy(data).cuda(), overlap, border).cpu().numpy()
    plan.check()
    ref = omfbd.half_spectrum(opatches.spectra_from_frames(data.astype(np.float64), n, overlap, border))
    err = np.abs(d - ref).max() / np.abs(ref).max()
    assert err <= 1e-5, err


@pytest.mark.parametrize("n_modes,diams,n_frames,n_patches", [
    (1, (31.0,), 1, 1), (8, (33.0, 20.0), 3, 5),   # one step of modes; odd boxes, one tile of units and pixels
    (25, (36.0,), 11, 12), (33, (28.0, 24.0), 12, 11),  # remainders in modes, units (132) and pixels
    (136, (32.0,), 4, 32),                          # a whole tile of units, modes beyond the tensor-core tiles
])
def test_simt_projection_edges(n_modes, diams, n_frames, n_patches):
    """The SIMT phase projection at the edges of its tiles and of its copies ahead, through the OTFs it leads to
    (within 2e-6 of the oracle's, as for the other OTFs)."""
    import numpy as np
    import torch

    from oracle import mfbd as omfbd
    case = cases.make_case(n_pix=64, diams=diams, wavelengths=(6563.0, 8542.0)[:len(diams)], n_frames=n_frames,
                           n_modes=n_modes, basis="zernike", n_patches=n_patches, seed=20250700 + n_modes)
    a32, _, _ = _inputs(case)
    plan = _plan_for(case, projection="simt")
    assert plan.info()["tc_projection"] == 0
    h = plan.otf(torch.from_numpy(a32).cuda()).cpu().numpy()
    for p in range(n_patches):
        for k, inter in enumerate(omfbd.otf_patch(case["setup"], a32[p].astype(np.float64))):
            assert np.abs(h[p, k] - omfbd.half_spectrum(inter["H"])).max() <= 2e-6, (p, k)
