"""The float-float amplitude generator in other units than GeV, where the
Breit-Wigner's denominator is large and its product with a small Y_l^m leaves the
range in which float pairs keep their low part: such amplitudes are FP64's.

As in test_gpu_ampgen_ff: both evaluations give the float nearest to the model's
value, one component in 10^6 may differ by FP64's own rounding.
"""
import numpy as np
import pytest

from test_gpu_ampgen_ff import agree, both, pwa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [1e3, 1e6, 3e7, 2e8])
def test_small_harmonics(pwa, unit):  # noqa: F811
    """l = m = 10 and 4 near the axis: |Y| from 1e-18 up, at every mass. (The widths
    keep (M Gamma)^2 below 2^80, above which everything is FP64's.)"""
    rng = np.random.default_rng(int(unit))
    n = 200_000
    s = 10.0 ** rng.uniform(-1.75, -0.3, n)           # sin(theta)
    kin = np.stack([unit * rng.uniform(0.98, 3.0, n), np.sqrt(1 - s * s), rng.uniform(0, 2 * np.pi, n)], axis=1)
    waves = [(unit * M, unit * G, l, m) for M, G in ((1.0, 1e-5), (2.9, 4e-6), (3.5, 2e-6))
             for l, m in ((10, 10), (10, -9), (4, 4))]
    agree(*both(pwa, waves, kin))
