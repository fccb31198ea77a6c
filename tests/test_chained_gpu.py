"""Chained launches (each kernel's set-up over its predecessor's tail) change no
bits: every kind of plan against its own captured graph, whose launches are not
chained, call after call; two plans at once on two streams against each alone;
and a batch that mixes pupils within and beyond half a patch against plans of
its problems (loss 1e-5 relative, dL/da and object 1e-4 norm-wise)."""

import numpy as np
import pytest
import torch

from tests import cases
from tests.test_parity_gpu import _inputs, _plan_for

pytestmark = pytest.mark.gpu

# n_pix, pupils, frames, patches, plan options
KINDS = [
    (64, (32.0,), 8, 1, {}),                                  # a cluster of CTAs per pair
    (64, (36.0, 28.0), 5, 90, {}),                            # one CTA per pair, more pairs than SMs
    (64, (36.0,), 12, 100, {}),                               # one CTA per pair, fewer
    (64, (36.0,), 15, 6, {}), (64, (44.0,), 3, 6, {}),        # general kernels
    (64, (30.0,), 4, 6, {"projection": "simt"}), (64, (30.0,), 4, 6, {"split": True}),
    (48, (20.0, 26.0), 3, 9, {}), (96, (40.0,), 4, 5, {}), (96, (40.0,), 4, 5, {"recompute": True}),
    (128, (56.0,), 3, 4, {}), (128, (70.0,), 20, 2, {"recompute": True}),
]


def _prepared(n_pix, diams, frames, patches, options):
    case = cases.make_case(n_pix=n_pix, diams=diams, wavelengths=(6563.0, 8542.0)[:len(diams)], n_frames=frames,
                           n_modes=12, basis="zernike", n_patches=2, seed=20251500 + n_pix + frames)
    a32, d32, _ = _inputs(case)
    reps = -(-patches // 2)
    a = torch.from_numpy(np.tile(a32, (reps, 1, 1))[:patches]).cuda()
    d = torch.from_numpy(np.tile(d32, (reps, 1, 1, 1, 1))[:patches]).cuda()
    return _plan_for(case, n_patches=patches, **options), a, d


@pytest.mark.parametrize("kind", KINDS)
def test_chained_calls_match_the_captured_graph(kind):
    plan, a, d = _prepared(*kind)
    loss, grad, obj = (torch.empty_like(t) for t in plan.loss_grad(a, d, want_object=True))
    graph = plan.capture(a, d, loss, grad, obj)
    graph.replay()
    for _ in range(5):
        out = plan.loss_grad(a, d, want_object=True)
        plan.check()
        for x, y in zip(out, (loss, grad, obj)):
            assert torch.equal(x, y)


@pytest.mark.parametrize("first,second", [(0, 2), (1, 7), (3, 8), (2, 10)])
def test_two_plans_on_two_streams(first, second):
    prepared = [_prepared(*KINDS[first]), _prepared(*KINDS[second])]
    alone = [p.loss_grad(a, d, want_object=True) for p, a, d in prepared]
    streams = [torch.cuda.Stream() for _ in prepared]
    torch.cuda.synchronize()
    outs = [[], []]
    for _ in range(8):
        for i, (p, a, d) in enumerate(prepared):
            with torch.cuda.stream(streams[i]):
                outs[i].append(p.loss_grad(a, d, want_object=True, stream=streams[i]))
    torch.cuda.synchronize()
    for i, (p, _, _) in enumerate(prepared):
        p.check()
        for out in outs[i]:
            for x, y in zip(out, alone[i]):
                assert torch.equal(x, y)


def test_batch_of_pupils_within_and_beyond_half_a_patch():
    from paper_2505_10639_gb300.mfbd import Batch, Plan, Problem
    shapes = [(n, f * n, j) for n in (48, 64, 96, 128) for f, j in ((0.375, 4), (0.5, 9), (0.5625, 3), (0.75, 17))]
    data = []
    for i, (n, diam, frames) in enumerate(shapes):
        case = cases.make_case(n_pix=n, diams=(diam,), wavelengths=(6563.0,), n_frames=frames, n_modes=9,
                               basis="zernike", n_patches=1, seed=20251600 + i)
        a32, d32, _ = _inputs(case)
        data.append((case, torch.from_numpy(a32).cuda(), torch.from_numpy(d32).cuda()))
    b = Batch([Problem(c["n_pix"], 1, c["diams"], c["wavelengths"], c["n_frames"], 9, gamma=c["setup"].gamma)
               for c, _, _ in data])
    out = b.loss_grad(Batch.pack([a for _, a, _ in data]), Batch.pack([d for _, _, d in data]), want_object=True)
    b.check()
    loss, grad, obj = (b.unpack(t, k) for t, k in zip(out, ("loss", "grad", "object")))
    for i, (c, a, d) in enumerate(data):
        plan = Plan(c["n_pix"], 1, list(c["diams"]), list(c["wavelengths"]), c["n_frames"], 9, basis="zernike",
                    gamma=c["setup"].gamma, projection="simt")
        lp, gp, op = plan.loss_grad(a, d, want_object=True)
        assert abs(loss[i].item() - lp.item()) <= 1e-5 * abs(lp.item()), shapes[i]
        assert (grad[i] - gp).norm().item() <= 1e-4 * gp.norm().item(), shapes[i]
        assert (obj[i] - op).abs().max().item() <= 1e-4 * op.abs().max().item(), shapes[i]
