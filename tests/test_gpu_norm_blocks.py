"""The tensor-core kernel of M beyond 20 waves: one launch up to 32 waves,
three launches over pairs of wave blocks beyond, and the 1024-event
accumulation period at its largest digit sums.

Tolerances as in test_gpu_norm (the digit bound of the sample, and 1e-12 of
the largest entry). The constant sample: every float is 127 (2^-7 + 2^-15 +
2^-23), digits 127, 127, 127, 0, 0 under r = 1, so each digit sum over a
period is 1024 * 127^2 = 1.65e7 quanta, just below 2^24; nothing is dropped,
and what remains are the float-float sums of 8 blocks over the CTA's periods
(two here), each within 2^-46 of the running sum, and ~150 FP64 additions:
16 * 2^-46 + 150 * 2^-53 < 2.5e-13. A lost quantum per digit sum would show at
2^-24 of it.
"""
import numpy as np
import pytest

import synth
from test_gpu_norm import build_M, digit_bound, oracle_M, pwa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n_mc", [(21, 64), (24, 1025), (25, 30001), (32, 155649), (32, 1),
                                    (33, 63), (36, 9729), (37, 20001), (41, 4097), (48, 65537)])
def test_norm_many_waves(pwa, N, n_mc):  # noqa: F811
    wl = synth.mixture_workload("n", synth.waves_linear(N), 10, n_mc, seed_mc=500 + N)
    M = build_M(pwa, wl.A_mc, wl.n_gen)
    Mo = oracle_M(wl.A_mc, wl.n_gen)
    err = np.abs(M - Mo)
    assert np.all(err <= digit_bound(wl.A_mc, wl.n_gen) + 1e-14 * np.abs(Mo).max())
    assert err.max() <= 1e-12 * np.abs(Mo).max(), err.max() / np.abs(Mo).max()
    assert np.array_equal(M, M.conj().T)
    assert np.array_equal(M, build_M(pwa, wl.A_mc, wl.n_gen)), "run-to-run bitwise"


@pytest.mark.parametrize("N", [4, 20, 24, 32, 48])
def test_norm_largest_digit_sums(pwa, N):  # noqa: F811
    n = 152 * 1024 * 2
    x = 127 * (2.0 ** -7 + 2.0 ** -15 + 2.0 ** -23)
    assert float(np.float32(x)) == x
    A = np.full((n, N), x, np.complex64)
    M = build_M(pwa, A, float(n))
    assert np.max(np.abs(M - x * x)) <= 2.5e-13 * x * x
