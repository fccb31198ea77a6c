"""The 6- and 12-point transforms of a lane (lines of 48 and 96 points) on the
host, against the definition in 64 bits. The error bounds lie between what the
prime-factor form has, which multiplies by no rounded twiddles (4.8e-8 to 5.1e-8
and 5.76e-8, with and without fused multiply-adds), and what three P-point
transforms with twiddles have (5.58e-8 to 5.62e-8 and 5.96e-8 to 6.24e-8)."""

import numpy as np
import pytest

from paper_2505_10639_gb300 import _lib


@pytest.mark.parametrize("kind,n,bound", [(9, 6, 5.35e-8), (10, 12, 5.85e-8)])
def test_lane_transform_error(kind, n, bound):
    lib = _lib.load()
    z = np.random.default_rng(5).standard_normal((20000, 2 * n)).astype(np.float32)
    out = np.empty_like(z)
    for x, y in zip(z, out):
        assert lib.mfbd_test_fft_host(kind, x.ctypes.data, y.ctypes.data) == 0
    k = np.arange(n)
    dft = np.exp(-2j * np.pi * (np.outer(k, k) % n) / n)
    ref = (z[:, 0::2].astype(np.float64) + 1j * z[:, 1::2]) @ dft
    got = out[:, 0::2].astype(np.float64) + 1j * out[:, 1::2]
    assert np.abs(got - ref).max() <= 2e-6 * np.abs(ref).max()
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err <= bound, err
