"""Uneven batches at the frame counts where the frame reduction changes its
form (8, 16 and 32 frames, one more each, and an odd split over two lanes):
every schedule and either kernel variant give the same bits, which agree with
the FP64 oracle within the tolerances of the FP32 path (loss 1e-5 relative,
dL/da and object 1e-4 norm-wise)."""

import pytest
import torch

from tests import cases
from tests.test_parity_gpu import _check, _inputs, _oracle

pytestmark = pytest.mark.gpu

# (n_pix, pupil, frames)
SHAPES = [(48, 20.0, 8), (64, 30.0, 9), (96, 40.0, 16), (48, 24.0, 17), (64, 28.0, 24), (48, 22.0, 32), (64, 32.0, 33),
          (128, 50.0, 13)]


@pytest.fixture(scope="module")
def problems():
    from paper_2505_10639_gb300.mfbd import Batch, Problem
    data = []
    for i, (n, diam, frames) in enumerate(SHAPES):
        case = cases.make_case(n_pix=n, diams=(diam,), wavelengths=(6563.0,), n_frames=frames, n_modes=6,
                               basis="zernike", n_patches=1, seed=20251100 + i)
        a32, d32, d_or = _inputs(case)
        data.append((case, a32, d32, _oracle(case, a32, d_or)))
    coeffs = Batch.pack([torch.from_numpy(a).cuda() for _, a, _, _ in data])
    spectra = Batch.pack([torch.from_numpy(d).cuda() for _, _, d, _ in data])
    probs = [Problem(c["n_pix"], 1, c["diams"], c["wavelengths"], c["n_frames"], c["n_modes"], gamma=c["setup"].gamma)
             for c, _, _, _ in data]
    return data, Batch(probs), coeffs, spectra


@pytest.mark.parametrize("mode", ["one_launch", "staged"])
@pytest.mark.parametrize("variant", [0, 1])
def test_every_schedule_and_variant_gives_the_same_bits(problems, mode, variant):
    data, b, coeffs, spectra = problems
    b.set_schedule("one_launch", 0, 0, 0)
    ref = b.loss_grad(coeffs, spectra, want_object=True)
    b.set_schedule(mode, 0, 0, variant)
    out = b.loss_grad(coeffs, spectra, want_object=True)
    b.check()
    for name, x, y in zip(("loss", "grad", "object"), out, ref):
        for i, (u, v) in enumerate(zip(b.unpack(x, name), b.unpack(y, name))):
            assert torch.equal(u, v), (name, SHAPES[i])
    loss, grad, obj = (b.unpack(t, k) for t, k in zip(out, ("loss", "grad", "object")))
    for i, (case, _, _, want) in enumerate(data):
        _check(case, loss[i].cpu().numpy(), grad[i].cpu().numpy(), obj[i].cpu().numpy().astype("complex128"), want)
