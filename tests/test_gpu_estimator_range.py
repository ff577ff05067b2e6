"""P(k) and bispectrum of FP32 fields whose measured modes lie far below the largest mode.

delta = 1 on every other plane (modes k = 0 and k_x = N/2 only) plus v = 2^-70 at one point of a plane
between them, which gives every other mode |delta_k| = v: P = box^3 v^2 / n^6 in every shell below
the Nyquist index, B = box^6 v^3 / n^9 and Q = n^3 / (3 v).  On power-of-two meshes the large values add and
cancel without rounding, so the FP32 transforms hold v everywhere else to their own rounding (1e-5, the bound of
the FP32 spectra elsewhere)."""
import math

import numpy as np
import pytest

from test_gpu_parity import OM
from test_gpu_parity import dgp, torch_dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu
V = 2.0 ** -70


def _field(torch, dev, n):
    d = torch.zeros((n, n, n), device=dev)
    d[::2] = 1.0
    d[1, 0, 0] = V
    return d


@pytest.mark.parametrize("n", [16, 32, 64, 128])
def test_power_of_shells_far_below_the_largest_mode(dgp, torch_dev, n):
    torch, dev = torch_dev
    box = 100.0
    ctx = dgp.dgp_init(box, n, 1.0, OM, precision=dgp.DGP_FP32)
    try:
        _, p, _ = dgp.power_spectrum(ctx, _field(torch, dev, n), n // 2 - 1)
    finally:
        dgp.dgp_destroy(ctx)
    assert np.allclose(p / (box ** 3 * V ** 2 / n ** 6), 1.0, rtol=0, atol=1e-5)


@pytest.mark.parametrize("n", [32, 64, 128])
def test_bispectrum_of_shells_far_below_the_largest_mode(dgp, torch_dev, n):
    torch, dev = torch_dev
    box = 100.0
    kf = 2 * math.pi / box
    ctx = dgp.dgp_init(box, n, 1.0, OM, precision=dgp.DGP_FP32)
    try:
        b, q = dgp.bispectrum(ctx, _field(torch, dev, n), 3 * kf, 4 * kf, [0.3, 1.2, 2.0])
    finally:
        dgp.dgp_destroy(ctx)
    assert np.allclose(b / (box ** 6 * V ** 3 / n ** 9), 1.0, rtol=0, atol=1e-5)
    assert np.allclose(q * V * 3 / n ** 3, 1.0, rtol=0, atol=1e-5)
