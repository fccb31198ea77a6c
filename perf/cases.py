"""Workloads a user of the package runs, as measurable cases.

Every case is one pass through the public entry points (``Plan``, ``Batch``,
``momfbd_loss``, ``dict_loss_grad``) on seeded synthetic data: granulation-like
objects (k^-3 power spectrum, contrast 10 %), Kolmogorov wavefronts, white
noise of 1e-3 of the mean. ``exact`` evaluates the same definitions with torch
in 64 bits: P = A exp(i phi), s = |F P|^2 / sum, H = F s, the Wiener object and
the object-eliminated loss, differentiated by autograd.

The library sums the loss in float64 from float32 terms; the programs here keep
it in float32, the type of the coefficients they optimise.
"""

import functools
import math
import random

import numpy as np
import torch

from paper_2505_10639_gb300.mfbd import Batch, Plan, Problem, dict_loss_grad, momfbd_loss

SIGMA = 1e-3


def listed():
    def field(name, kind, n_pix, rows, cols, overlap, diams, frames, modes, basis="kl", d_r0=5.0, precision="fp32",
              recompute=False):
        return dict(name=name, kind=kind, n_pix=n_pix, rows=rows, cols=cols, overlap=overlap, diams=diams,
                    frames=frames, modes=modes, basis=basis, d_r0=d_r0, precision=precision, recompute=recompute)

    return [
        # One patch, one object, a short burst: an interactive check or a quick look at one star or pore.
        field("single_64px", "loss_grad", 64, 1, 1, 32, "32", 8, 20, basis="zernike"),
        # One optimiser step over a 1024 x 1024 field, wideband and narrowband, through autograd.
        field("field_64px_autograd", "autograd", 64, 31, 31, 32, "36,28", 12, 44),
        # One step over a 512 x 512 field with longer bursts (15 frames of two cameras).
        field("field_64px_15frames", "loss_grad", 64, 15, 15, 32, "36,28", 15, 54),
        # Larger patches over a 512 x 512 field, closely spaced (96 px every 40), two cameras, 12 frames.
        field("field_96px", "loss_grad", 96, 11, 11, 56, "48,38", 12, 54),
        # 128 px patches over a 512 x 512 field, one camera, 15 frames, FP32.
        field("field_128px_1object", "loss_grad", 128, 7, 7, 64, "56", 15, 54),
        # A quarter of a 4096 x 4096 field: four wavelengths, 32 frames, 100 modes, BF16 phases, the field
        # recomputed in the backward pass to save memory.
        field("field_128px_4objects", "loss_grad", 128, 31, 31, 64, "40,48,56,64", 32, 100, d_r0=10.0,
              precision="bf16_phase", recompute=True),
        # Many unlike problems at once (every patch size, 1 to 3 objects, 8 to 24 frames), one launch.
        dict(name="batch_uneven", kind="batch", problems=500, layout=20250518),
        # The object-inferring loss: gradients in the coefficients and in the objects.
        field("explicit_64px", "explicit", 64, 15, 15, 32, "36,28", 12, 44),
        # The spatially variant model on a PSF dictionary: gradients in the object and the coefficient maps.
        dict(name="dictionary_64px", kind="dictionary", patches=225, objects=2, frames=12, atoms=8),
        # From camera frames to patch spectra, before the optimisation.
        field("spectra_64px", "spectra", 64, 31, 31, 32, "36,28", 12, 44),
        # After the optimisation of a long burst (100 frames): loss, objects, filter, mosaic.
        field("restore_64px_100frames", "restore", 64, 15, 15, 32, "32", 100, 135),
        # The noise filter of the objects from the data and the OTFs.
        field("noise_filter_64px", "noise_filter", 64, 31, 31, 32, "36,28", 12, 44),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loss_grad"] * 4 + ["autograd", "explicit", "restore", "spectra", "noise_filter", "batch",
                                           "dictionary"])
    if kind == "batch":
        return dict(kind=kind, problems=_log_int(rng, 4, 600), layout=rng.randrange(1 << 30))
    if kind == "dictionary":
        return dict(kind=kind, patches=_log_int(rng, 1, 300), objects=rng.randint(1, 3), frames=rng.randint(1, 16),
                    atoms=rng.randint(2, 12))
    n = rng.choice([48, 64, 64, 96, 128])
    objects, frames = rng.randint(1, 4), _log_int(rng, 2, 40)
    most = 900000 * (64 * 64) // (n * n * objects * frames)  # no more than the largest listed case
    patches = _log_int(rng, 1, max(1, min(961, most)))
    rows = max(1, int(math.sqrt(patches) * rng.uniform(0.6, 1.0)))
    lo, hi = math.ceil(0.35 * n), n // 2
    return dict(kind=kind, n_pix=n, rows=rows, cols=max(1, patches // rows), overlap=rng.choice([n // 2, n // 4, n // 2 + 3]),
                diams=",".join(str(rng.choice([rng.randint(lo, hi), 2 * rng.randint((lo + 1) // 2, hi // 2)]))
                               for _ in range(objects)),
                frames=frames, modes=_log_int(rng, 20, 135), basis=rng.choice(["kl", "zernike"]),
                d_r0=rng.choice([3.0, 5.0, 10.0]),
                precision=rng.choice(["fp32", "fp32", "bf16_phase"]), recompute=n > 64 and rng.random() < 0.5)


# ------------------------------------------------------------------ optics

def _noll(j):
    n = 0
    while (n + 1) * (n + 2) // 2 < j:
        n += 1
    p = j - n * (n + 1) // 2 - 1
    return n, (2 * ((p + 1) // 2) if n % 2 == 0 else 2 * (p // 2) + 1)


def _covariance(count):
    """Kolmogorov covariance of the Zernike coefficients 2..count + 1, in units of (D/r0)^(5/3)."""
    g = math.gamma
    mu = 8 / 3
    radial = -g((1 - mu) / 2) / (2 ** mu * g((1 + mu) / 2))
    a = 2 * (24 / 5 * g(6 / 5)) ** (5 / 6) / (4 * math.pi * (2 * math.pi) ** (5 / 3) * radial)
    k = a * 8 * math.pi ** (8 / 3) * g(14 / 3) / 2 ** (14 / 3)
    nm = [_noll(j) for j in range(2, count + 2)]
    cov = np.zeros((count, count))
    for u, (n, m) in enumerate(nm):
        for v, (n2, m2) in enumerate(nm):
            if m == m2 and (m == 0 or u % 2 == v % 2):
                # both arguments are positive, and their gammas overflow at high orders
                num, den = (n + n2 - 5 / 3) / 2, (n + n2 + 23 / 3) / 2
                ratio = math.exp(math.lgamma(num) - math.lgamma(den))
                cov[u, v] = (k * (-1) ** ((n + n2 - 2 * m) // 2) * math.sqrt((n + 1) * (n2 + 1)) * ratio
                             / (g((n - n2 + 17 / 3) / 2) * g((n2 - n + 17 / 3) / 2)))
    return cov, nm


@functools.lru_cache(maxsize=None)
def _modes(basis, count):
    """(coefficients on Zernike 2.., variances) of the modes."""
    if basis == "zernike":
        cov, _ = _covariance(count)
        return np.eye(count), np.diag(cov).copy()
    n = 0
    while (n + 1) * (n + 2) // 2 < 4 * count + 1:
        n += 1
    total = (n + 1) * (n + 2) // 2 - 1
    cov, nm = _covariance(total)
    groups = {}
    for i, (_, m) in enumerate(nm):
        groups.setdefault((m, 0 if m == 0 else i % 2), []).append(i)  # index 0 is Noll 2: even i, cosine
    found = []
    for (m, sine), at in groups.items():
        values, vectors = np.linalg.eigh(cov[np.ix_(at, at)])
        for value, vector in zip(values, vectors.T):
            row = np.zeros(total)
            row[at] = vector * np.sign(vector[np.argmax(np.abs(vector))])
            found.append((-float("%.9e" % value), m, sine, row, value))
    found.sort(key=lambda f: f[:3])
    return np.array([f[3] for f in found[:count]]), np.array([f[4] for f in found[:count]])


@functools.lru_cache(maxsize=None)
def _pupil(n_pix, diam, basis, count):
    """(pupil pixels as flat indices, modes [count, pixels]) of a diam px pupil on an n_pix grid."""
    c = (n_pix - 1) / 2
    y, x = np.mgrid[0:n_pix, 0:n_pix] - c
    inside = x * x + y * y <= diam * diam / 4
    rho, theta = (np.hypot(x, y) / (diam / 2))[inside], np.arctan2(y, x)[inside]
    mix, _ = _modes(basis, count)
    zernike = []
    for j in range(2, mix.shape[1] + 2):
        n, m = _noll(j)
        radial = sum((-1) ** s * math.factorial(n - s) / (math.factorial(s) * math.factorial((n + m) // 2 - s)
                     * math.factorial((n - m) // 2 - s)) * rho ** (n - 2 * s) for s in range((n - m) // 2 + 1))
        angle = 1.0 if m == 0 else math.sqrt(2) * (np.cos(m * theta) if j % 2 == 0 else np.sin(m * theta))
        zernike.append(math.sqrt(n + 1) * radial * angle)
    out = mix @ np.array(zernike)
    if basis == "kl":  # orthonormal on the sampled pupil, in order
        for i in range(count):
            for p in range(i):
                out[i] -= (out[p] @ out[i] / rho.size) * out[p]
            out[i] /= math.sqrt(out[i] @ out[i] / rho.size)
    return np.flatnonzero(inside), out


class _Optics:
    """Forward model of one object in torch, any precision."""

    def __init__(self, n_pix, diam, scale, basis, count, dtype):
        at, modes = _pupil(n_pix, diam, basis, count)
        self.n, self.at = n_pix, torch.from_numpy(at).cuda()
        self.modes = torch.from_numpy(modes).cuda().to(dtype) * scale

    def phases(self, a):
        return a @ self.modes

    def otf(self, phases):
        p = torch.zeros(phases.shape[:-1] + (self.n * self.n,), dtype=phases.dtype, device=phases.device)
        p = torch.complex(p.index_copy(-1, self.at, torch.cos(phases)), p.index_copy(-1, self.at, torch.sin(phases)))
        s = torch.fft.fft2(p.unflatten(-1, (self.n, self.n))).abs().square()
        return torch.fft.rfft2(s / s.sum((-2, -1), keepdim=True))


# ------------------------------------------------------------------ inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _object_field(g, shape):
    h, w = shape[-2:]
    k = torch.hypot(torch.fft.fftfreq(h, device="cuda")[:, None], torch.fft.fftfreq(w, device="cuda")[None, :])
    amp = torch.where(k > 0, k.clamp_min(1e-9) ** -1.5, 0.0)
    f = torch.fft.ifft2(torch.randn(shape, generator=g, device="cuda", dtype=torch.complex64) * amp).real
    f = (f - f.mean((-2, -1), keepdim=True)) / f.std((-2, -1), keepdim=True)
    return (1.0 + 0.1 * f).clamp_min(1e-3)


def _diams(case):
    return [float(d) for d in case["diams"].split(",")]


def _field_size(case):
    n, stride = case["n_pix"], case["n_pix"] - case["overlap"]
    return (case["rows"] - 1) * stride + n, (case["cols"] - 1) * stride + n


def _wavelengths(diams):
    return [6563.0 * diams[0] / d for d in diams]


def _gamma(n_pix):
    return 1e-3 * n_pix * n_pix * SIGMA * SIGMA


def _problem_data(g, n, diams, frames, modes, basis, d_r0, objects):
    """Coefficients [P, J, M] and spectra [P, K, J, n, n/2+1] of the patch objects [P, K, n, n]."""
    patches = objects.shape[0]
    spread = torch.from_numpy(np.sqrt(_modes(basis, modes)[1] * d_r0 ** (5 / 3))).cuda().float()
    true, off = (torch.randn((patches, frames, modes), generator=g, device="cuda") * spread for _ in range(2))
    spectra = torch.empty((patches, len(diams), frames, n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    chunk = max(1, (1 << 24) // (frames * n * n))
    for k, d in enumerate(diams):
        optics = _Optics(n, d, d / diams[0], basis, modes, torch.float32)
        for p in range(0, patches, chunk):
            o = torch.fft.rfft2(objects[p:p + chunk, k])
            noise = torch.randn((o.shape[0], frames, n, n), generator=g, device="cuda") * SIGMA
            spectra[p:p + chunk, k] = o[:, None] * optics.otf(optics.phases(true[p:p + chunk])) + torch.fft.rfft2(noise)
    return true + 0.3 * off, spectra


def _field_data(case, seed):
    g = _generator(seed)
    n, diams, stride = case["n_pix"], _diams(case), case["n_pix"] - case["overlap"]
    field = _object_field(g, (len(diams),) + _field_size(case))
    patches = field.unfold(1, n, stride).unfold(2, n, stride).flatten(1, 2).transpose(0, 1).contiguous()
    return _problem_data(g, n, diams, case["frames"], case["modes"], case["basis"], case["d_r0"], patches)


def _frames_data(case, seed):
    g = _generator(seed)
    shape = _field_size(case)
    field = _object_field(g, (len(_diams(case)), 1) + shape)
    return field + SIGMA * torch.randn((field.shape[0], case["frames"]) + shape, generator=g, device="cuda")


def _layout(case):
    """The problems of an uneven batch: sizes from {48, 64, 96, 128}, 1-3 objects, 8-24 frames, 20-66 modes."""
    r = random.Random(case["layout"])
    out = []
    for _ in range(case["problems"]):
        n = r.choice([48, 64, 96, 128])
        diams = [2.0 * round(r.uniform(0.35, 0.5) * n / 2) for _ in range(r.randint(1, 3))]
        out.append((n, diams, r.randint(8, 24), r.randint(20, 66)))
    return out


def _batch_data(case, seed):
    g = _generator(seed)
    return [_problem_data(g, n, diams, frames, modes, "zernike", 5.0, _object_field(g, (1, len(diams), n, n)))
            for n, diams, frames, modes in _layout(case)]


def _dictionary_data(case, seed):
    g = _generator(seed)
    p, k, j, m, n = case["patches"], case["objects"], case["frames"], case["atoms"], 64
    width, centre = (torch.rand((2, m, 2), generator=g, device="cuda"))
    x = torch.arange(n, device="cuda")
    d = (x - (3 * centre[..., None] - 1.5)).abs()
    d = torch.exp(-0.5 * (torch.minimum(d, n - d) / (0.8 + 3.2 * width[..., None])) ** 2)
    atoms = d[:, 0, :, None] * d[:, 1, None, :]
    atom_otf = torch.fft.rfft2(atoms / atoms.sum((-2, -1), keepdim=True))
    coeff = 0.1 + torch.rand((p, k, j, m, n, n), generator=g, device="cuda")
    coeff /= coeff.sum(3, keepdim=True)
    obj = _object_field(g, (p, k, n, n))
    noise = SIGMA * torch.randn((p, k, j, n, n), generator=g, device="cuda")
    blurred = torch.fft.rfft2(_object_field(g, (p, k, n, n))) * atom_otf.mean(0)
    spectra = blurred[:, :, None] + torch.fft.rfft2(noise)
    gamma = torch.full((k, j), 1.0 / j, device="cuda")
    return atom_otf.contiguous(), gamma, obj, coeff, spectra


# ------------------------------------------------------------------- cases

def _plan(case):
    diams = _diams(case)
    return Plan(case["n_pix"], case["rows"] * case["cols"], diams, _wavelengths(diams), case["frames"], case["modes"],
                basis=case["basis"], gamma=_gamma(case["n_pix"]), precision=case["precision"],
                recompute=case["recompute"])


def prepare(case, seed):
    s = dict(case=case)
    kind = case["kind"]
    if kind == "batch":
        layout, data = _layout(case), _batch_data(case, seed)
        s["batch"] = Batch([Problem(n, 1, diams, _wavelengths(diams), frames, modes, gamma=_gamma(n))
                            for n, diams, frames, modes in layout])
        s["coeffs"], s["spectra"] = Batch.pack([d[0] for d in data]), Batch.pack([d[1] for d in data])
        loss, grad, _ = s["batch"].outputs()
        s["batch"].autotune(s["coeffs"], s["spectra"], loss, grad, reps=1)
        return s
    if kind == "dictionary":
        s["inputs"] = _dictionary_data(case, seed)
        return s
    s["plan"] = _plan(case)
    if kind == "spectra":
        s["frames"] = _frames_data(case, seed)
        return s
    s["coeffs"], s["spectra"] = _field_data(case, seed)
    if kind == "autograd":
        s["coeffs"].requires_grad_()
    elif kind == "explicit":  # the first object of an object-inferring run: the average frame
        s["object"] = s["spectra"].mean(2)
    elif kind == "noise_filter":
        s["otf"], s["object"] = _otf(case, s["coeffs"]), s["spectra"].mean(2)
    return s


def _otf(case, a):
    """The OTFs at the coefficients, in float32, with torch."""
    diams, n = _diams(case), case["n_pix"]
    out = torch.empty((a.shape[0], len(diams), a.shape[1], n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    chunk = max(1, (1 << 24) // (a.shape[1] * n * n))
    for k, d in enumerate(diams):
        optics = _Optics(n, d, d / diams[0], case["basis"], case["modes"], torch.float32)
        for p in range(0, a.shape[0], chunk):
            out[p:p + chunk, k] = optics.otf(optics.phases(a[p:p + chunk]))
    return out


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "loss_grad":
        loss, grad, obj = s["plan"].loss_grad(s["coeffs"], s["spectra"], want_object=True)
        return loss.float(), grad, obj
    if kind == "autograd":
        loss = momfbd_loss(s["coeffs"], s["spectra"], s["plan"])
        (grad,) = torch.autograd.grad(loss.sum(), s["coeffs"])
        return loss.detach().float(), grad
    if kind == "explicit":
        loss, grad, grad_obj = s["plan"].loss_grad_explicit(s["coeffs"], s["spectra"], s["object"])
        return loss.float(), grad, grad_obj
    if kind == "batch":
        loss, grad, obj = s["batch"].loss_grad(s["coeffs"], s["spectra"], want_object=True)
        return loss.float(), grad, obj
    if kind == "dictionary":
        loss, grad_obj, grad_coeff = dict_loss_grad(*s["inputs"])
        return loss.float(), grad_obj, grad_coeff
    if kind == "spectra":
        return s["plan"].spectra_from_frames(s["frames"], case["overlap"], case["n_pix"] // 8)
    if kind == "noise_filter":
        obj = s["object"].clone()
        return s["plan"].ls_filter_objects(s["spectra"], s["otf"], _noise_power(case), obj=obj), obj
    # restore
    loss, obj = s["plan"].forward(s["coeffs"], s["spectra"])
    s["plan"].filter_objects(obj, 0.75, 0.8)
    h, w = _field_size(case)
    return loss.float(), obj, s["plan"].merge_objects(obj, h, w, case["overlap"], case["n_pix"] // 8)


def _noise_power(case):
    return case["n_pix"] ** 2 * SIGMA ** 2


# -------------------------------------------------------------------- work

def _unit_flops(n, diams, modes, forward_only=False):
    """Operations of the path per (patch, frame), all objects: per object the transforms of the pupil's W columns,
    n field rows and two half-sized real transforms each way, the frame sums and the modal products."""
    total = 0.0
    for d in diams:
        pixels = math.pi / 4 * d * d
        line = 5.0 * n * math.log2(n)
        one_way = (d + 2 * n) * line + 2.0 * pixels * modes + 18.0 * n * (n // 2 + 1)
        total += one_way * (1 if forward_only else 2)
    return total


def work(case):
    kind = case["kind"]
    if kind == "batch":
        size = flops = 0.0
        for n, diams, frames, modes in _layout(case):
            half = 8.0 * n * (n // 2 + 1)
            size += 8.0 * frames * modes + (frames + 1) * len(diams) * half + 8
            flops += frames * _unit_flops(n, diams, modes)
        return {"bytes": size, "flops": flops}
    if kind == "dictionary":
        n, units = 64, case["patches"] * case["objects"] * case["frames"]
        maps, half = 4.0 * n * n, 8.0 * n * (n // 2 + 1)
        size = units * (2 * case["atoms"] * maps + half) + 2 * case["patches"] * case["objects"] * maps
        return {"bytes": size, "flops": units * 2.0 * case["atoms"] * n * 5 * n * math.log2(n)}
    n, diams, frames, modes = case["n_pix"], _diams(case), case["frames"], case["modes"]
    patches, half = case["rows"] * case["cols"], 8.0 * n * (n // 2 + 1)
    data, objects = patches * len(diams) * frames * half, patches * len(diams) * half
    h, w = _field_size(case)
    if kind == "spectra":
        return {"bytes": 4.0 * len(diams) * frames * h * w + data,
                "flops": patches * len(diams) * frames * n * 5.0 * n * math.log2(n)}
    if kind == "noise_filter":
        return {"bytes": 2 * data + 2.5 * objects, "flops": 2.0 * data}
    size = 4.0 * patches * frames * modes + data + 8 * patches
    if kind == "restore":
        return {"bytes": size + objects + 4.0 * len(diams) * h * w,
                "flops": patches * (frames * _unit_flops(n, diams, modes, True)
                                    + len(diams) * n * 5.0 * n * math.log2(n))}
    size += 4.0 * patches * frames * modes
    size += objects * {"loss_grad": 1, "autograd": 0, "explicit": 2}[kind]
    return {"bytes": size, "flops": patches * frames * _unit_flops(n, diams, modes)}


# ------------------------------------------------------------------- exact

def _plane(n):
    """How often each half-spectrum column stands in the full plane."""
    w = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0
    return w


def _exact_problem(n, diams, modes, basis, gamma, coeffs, spectra, precision, objects=None):
    """loss [P], dL/da, and the Wiener objects (or, for given objects, dL/dconj(O)) in 64 bits."""
    weight = _plane(n)
    total = torch.zeros(coeffs.shape[0], dtype=torch.float64, device="cuda")
    grads = torch.zeros(coeffs.shape, dtype=torch.float64, device="cuda")
    objs = torch.zeros(spectra.shape[:2] + spectra.shape[3:], dtype=torch.complex128, device="cuda")
    if precision == "bf16_phase":
        coeffs = coeffs.bfloat16()
    chunk = max(1, (1 << 23) // (coeffs.shape[1] * n * n))
    for k, diam in enumerate(diams):
        optics = _Optics(n, diam, 1.0, basis, modes, torch.float64)
        modes64 = optics.modes
        if precision == "bf16_phase":  # the operands of the product, as the entry point's option rounds them
            optics.modes = optics.modes.float().bfloat16().double()
        for p in range(0, coeffs.shape[0], chunk):
            phases = (optics.phases(coeffs[p:p + chunk].double()) * (diam / diams[0])).requires_grad_()
            d = spectra[p:p + chunk, k].to(torch.complex128)
            otf = optics.otf(phases)
            if objects is None:
                num, den = (d * otf.conj()).sum(1), otf.abs().square().sum(1) + gamma
                loss = ((d.abs().square().sum(1) - num.abs().square() / den) * weight).sum((-2, -1))
                objs[p:p + chunk, k] = (num / den).detach()
            else:
                o = objects[p:p + chunk, k].to(torch.complex128)
                r = d - o[:, None] * otf
                loss = ((r.abs().square().sum(1) + gamma * o.abs().square()) * weight).sum((-2, -1))
                objs[p:p + chunk, k] = (gamma * o - (otf.conj() * r).sum(1)).detach()
            total[p:p + chunk] += loss.detach()
            (g,) = torch.autograd.grad(loss.sum(), phases)
            grads[p:p + chunk] += g @ modes64.T * (diam / diams[0])
    return total, grads, objs


def _window(n, border):
    x = torch.arange(n, dtype=torch.float64, device="cuda") + 0.5
    x = torch.minimum(x, n - x)
    w = torch.where(x < border, 0.5 * (1 - torch.cos(math.pi * x / border)), 1.0)
    return w[:, None] * w[None, :]


def _exact_spectra(case, seed):
    frames = _frames_data(case, seed)
    n, stride = case["n_pix"], case["n_pix"] - case["overlap"]
    units = frames.unfold(2, n, stride).unfold(3, n, stride).flatten(2, 3).permute(2, 0, 1, 3, 4)
    window = _window(n, n // 8)
    out = []
    for patch in units.split(16):
        patch = patch.double()
        mean = patch.mean((-2, -1), keepdim=True)
        out.append(torch.fft.rfft2((patch - mean) * window + mean))
    return torch.cat(out)


def _exact_restore(case, seed):
    n, diams = case["n_pix"], _diams(case)
    coeffs, spectra = _field_data(case, seed)
    loss, _, obj = _exact_problem(n, diams, case["modes"], case["basis"], _gamma(n), coeffs, spectra,
                                  case["precision"])
    ky, kx = torch.fft.fftfreq(n, 1 / n).cuda().double(), torch.arange(n // 2 + 1, device="cuda").double()
    lo, hi = np.float32(0.75).item(), np.float32(0.8).item()
    for k, d in enumerate(diams):
        f = torch.hypot(ky[:, None], kx[None, :]) / d
        cosine = 0.5 * (1 + torch.cos(math.pi * (f - lo) / (hi - lo)))
        obj[:, k] *= torch.where(f <= lo, 1.0, torch.where(f >= hi, 0.0, cosine))
    h, w = _field_size(case)
    image = torch.fft.irfft2(obj, s=(n, n))
    window, stride = _window(n, n // 8), n - case["overlap"]
    total = torch.zeros((len(diams), h, w), dtype=torch.float64, device="cuda")
    cover = torch.zeros((h, w), dtype=torch.float64, device="cuda")
    for p in range(image.shape[0]):
        y, x = p // case["cols"] * stride, p % case["cols"] * stride
        total[:, y:y + n, x:x + n] += image[p] * window
        cover[y:y + n, x:x + n] += window
    return loss, obj, torch.where(cover > 0, total / cover.clamp_min(1e-300), 0.0)


def _exact_dictionary(case, seed):
    atom_otf, gamma, obj, coeff, spectra = _dictionary_data(case, seed)
    atom_otf, gamma, weight = atom_otf.to(torch.complex128), gamma.double(), _plane(64)
    loss = torch.zeros(case["patches"], dtype=torch.float64, device="cuda")
    grad_obj, grad_coeff = torch.empty(obj.shape, dtype=torch.float64, device="cuda"), []
    for p in range(case["patches"]):
        o, a = obj[p].double().requires_grad_(), coeff[p].double().requires_grad_()
        model = (torch.fft.rfft2(o[:, None, None] * a) * atom_otf).sum(2)
        r = (spectra[p].to(torch.complex128) - model).abs().square()
        loss[p] = one = ((r * weight).sum((-2, -1)) * gamma).sum()
        grad_obj[p], g = torch.autograd.grad(one, (o, a))
        grad_coeff.append(g.float() if case["patches"] * a.numel() > 1 << 28 else g)
    return loss.detach(), grad_obj, torch.stack(grad_coeff)


def exact(case, seed):
    kind = case["kind"]
    if kind == "noise_filter":  # a threshold, a median and a connected component: decisions, no computed number
        return None
    if kind == "spectra":
        return _exact_spectra(case, seed)
    if kind == "restore":
        return _exact_restore(case, seed)
    if kind == "dictionary":
        return _exact_dictionary(case, seed)
    if kind == "batch":
        got = [_exact_problem(n, diams, modes, "zernike", _gamma(n), a, d, "fp32")
               for (n, diams, _, modes), (a, d) in zip(_layout(case), _batch_data(case, seed))]
        return tuple(torch.cat([g[i].reshape(-1) for g in got]) for i in range(3))
    n = case["n_pix"]
    coeffs, spectra = _field_data(case, seed)
    loss, grad, obj = _exact_problem(n, _diams(case), case["modes"], case["basis"], _gamma(n), coeffs, spectra,
                                     case["precision"], spectra.mean(2) if kind == "explicit" else None)
    return (loss, grad) if kind == "autograd" else (loss, grad, obj)
