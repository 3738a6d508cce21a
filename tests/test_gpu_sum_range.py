"""The sums over CTAs keep the range of the FP32 sums that they are made of: the
Hessian beyond 20 waves, where V or the amplitudes are so large or small that totals
come near, or leave, what a float holds. Scaling V by 2^k scales every float of the
evaluation, and so H by 2^-2k, exactly until a float under- or overflows.
"""
import numpy as np
import pytest

from test_gpu_norm import pwa  # noqa: F401

pytestmark = pytest.mark.gpu


def amplitudes(n, N, big, seed):
    """Wave 0 large and of constant size: |S| varies little, no event stands out."""
    rng = np.random.default_rng(seed)
    A = (rng.standard_normal((n, N)) + 1j * rng.standard_normal((n, N))).astype(np.complex64)
    A[:, 0] = (big * np.exp(2j * np.pi * rng.random(n))).astype(np.complex64)
    return A


@pytest.mark.parametrize("N", [21, 24, 29, 32, 40, 48])
@pytest.mark.parametrize("k", [54, -57])
def test_hessian(pwa, N, k):  # noqa: F811
    """k = 54: sums near 2^-108 keep their low words (a product's rounding is at most
    2^-150, n of them 2^(2k - 150) n after scaling back; float pairs 2^-40 of
    sqrt(H_aa H_bb) with a wide margin). k = -57: every thread's sum is below 2^127
    (64 events of J^2 <= 2.2^2 2^114), the total of 20 000 above 2^128."""
    n = 20_000
    A = amplitudes(n, N, 400.0, N)
    V = np.ones(N, complex)
    with pwa.Likelihood(N) as L:
        L.load_events(A, A[:100], 100.0)
        H0, H = L.hessian(V), L.hessian(V * 2.0 ** k)
    if k < 0:
        assert H.max() > 2.0 ** 128
    assert np.all(np.isfinite(H))
    d = np.sqrt(np.diag(H0))
    err = np.abs(H * 2.0 ** (2 * k) - H0)
    assert np.all(err <= 2 * n * 2.0 ** (2 * max(k, 0) - 150) + 2.0 ** -40 * np.outer(d, d)), (err / np.outer(d, d)).max()
