"""The sums over CTAs keep the range of the FP32 sums that they are made of: the
Hessian beyond 20 waves and the gradients of the free-resonance form, where V or
the amplitudes are so large or small that totals come near, or leave, what a float
holds. Scaling V by 2^k scales every float of the evaluation, and so H by 2^-2k and
the gradient by 2^-k, exactly until a float under- or overflows.
"""
from types import SimpleNamespace

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


def res_sample(n, N, R, seed):
    A = np.roll(amplitudes(n, N, 400.0, seed), R, axis=1)     # the large wave is the first fixed one
    rng = np.random.default_rng(seed + 1)
    return rng.uniform(0.98, 3.0, n), A[:, :R].copy(), A[:, R:].copy()


@pytest.mark.parametrize("N,R", [(4, 1), (20, 4), (32, 8)])
def test_free_resonances(pwa, N, R):  # noqa: F811
    """The gradient in V of amplitudes of 2^60 at V of 2^-114: each warp's sum is a
    float (64 events a tile, 2^114 each, 10 tiles), the total of 400 000 events 2^132.
    The fixed waves' first one is large."""
    n = 400_000
    m, Y, A = res_sample(n, N, R, N)
    M, G = 1.0 + 0.2 * np.arange(R), np.full(R, 0.2)
    V = np.ones(N, complex)
    one = np.float32(2.0 ** 60)

    def load(s):    # one MC event of no weight to speak of (its term is I / n_gen)
        return SimpleNamespace(n_free=R, m_data=m, Y_data=Y * s, Afix_data=A * s, m_mc=m[:1],
                               Y_mc=Y[:1], Afix_mc=A[:1], n_gen=1e30)

    with pwa.Likelihood(N) as L:
        L.load_resonance_events(load(1))
        nll0, gV0, gM0, gW0 = L.nll_grad_res(V, M, G)
        L.load_resonance_events(load(one))
        nll, gV, gM, gW = L.nll_grad_res(V * 2.0 ** -114, M, G)
    assert np.abs(gV).max() > 2.0 ** 128
    assert np.all(np.isfinite(gV)) and np.all(np.isfinite(gM)) and np.all(np.isfinite(gW))
    size = np.abs(gV0).max()
    assert np.max(np.abs(gV * 2.0 ** -114 - gV0)) <= 1e-6 * size
    assert abs((nll - n * 2 * 54 * np.log(2)) - nll0) <= 1e-9 * abs(nll)
