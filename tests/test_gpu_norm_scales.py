"""M of samples whose amplitudes are far from 1 in size (other units, narrow
resonances: 1 / (M Gamma) is 1e-17 where M and Gamma are in eV): the digits of the
tensor-core kernel follow each wave's own scale, at any size.

The kernel's error per event and real entry of G is 2^-41 (|x_p| 2^r_q [|x_q| <
2^(r_q - 17)] + |x_q| 2^r_p [|x_p| < 2^(r_p - 17)]) + 2^(r_p + r_q - 61), r = the
exponent of the wave's largest |Re| + |Im| plus 2, whatever r is; M is held to that
bound computed from the sample, and to 1e-12 of sqrt(M_aa M_bb). Scaling waves by
powers of two scales the digits, their sums and M exactly.
"""
import numpy as np
import pytest

import oracle
from test_gpu_norm import build_M, pwa  # noqa: F401

pytestmark = pytest.mark.gpu


def bound(A, n_gen):
    X = np.empty((A.shape[0], 2 * A.shape[1]), np.float64)
    X[:, 0::2] = A.real
    X[:, 1::2] = A.imag
    amax = (np.abs(A.real) + np.abs(A.imag)).max(axis=0).astype(np.float64)
    r = np.repeat(np.where(amax > 0, np.floor(np.log2(np.where(amax > 0, amax, 1.0))) + 2, 0), 2)
    s, ax = 2.0 ** r, np.abs(X)
    small = (ax < 2.0 ** (r - 17)).astype(np.float64)
    B = 2.0 ** -41 * ((ax.T @ small) * s[None, :] + (small.T @ ax) * s[:, None]) \
        + 2.0 ** -61 * A.shape[0] * np.outer(s, s)
    return (B[0::2, 0::2] + B[1::2, 1::2] + B[0::2, 1::2] + B[1::2, 0::2]) / n_gen


def sample(N, n, seed=3):
    rng = np.random.default_rng(seed)
    m = rng.uniform(0.98, 3.0, n)
    out = np.empty((n, N), np.complex64)
    for a in range(N):
        M, G = 1.0 + 1.9 * a / N, 0.05 + 0.01 * (a % 7)
        out[:, a] = np.exp(2j * np.pi * (a % 3) * rng.random(n)) / (M * M - m * m - 1j * M * G)
    return out


@pytest.mark.parametrize("N", [3, 8, 16, 20, 24, 32, 41, 48])
@pytest.mark.parametrize("e", [-95, -60, -45, -38, 20, 60, 95])
def test_every_scale(pwa, N, e):  # noqa: F811
    n = 5000
    A = sample(N, n)
    B = A.copy()
    B[:, ::2] *= np.float32(2.0 ** e)       # every other wave; exact
    M0, M = build_M(pwa, A, 1.5 * n), build_M(pwa, B, 1.5 * n)
    s = np.where(np.arange(N) % 2 == 0, 2.0 ** e, 1.0)
    Mo = oracle.norm_matrix(B, 1.5 * n)
    d = np.sqrt(np.diag(Mo).real)
    err = np.abs(M - Mo)
    assert np.all(err <= bound(B, 1.5 * n) + 1e-14 * np.outer(d, d))
    assert np.max(err / np.outer(d, d)) <= 1e-12
    if e < 50:      # the same digits (beyond, the FP64 kernel serves the sample)
        assert np.array_equal(M / np.outer(s, s), M0)


@pytest.mark.parametrize("N", [8, 24, 41])
@pytest.mark.parametrize("scale", [2.0 ** -120, 1e-44, 2.0 ** 125])
def test_ends_of_the_float_range(pwa, N, scale):  # noqa: F811
    """Amplitudes near the smallest normal and subnormal floats and the largest ones."""
    n = 3000
    A = sample(N, n, 5)
    A[:, N // 2] = (A[:, N // 2].astype(np.complex128) * (scale / np.abs(A[:, N // 2]).max())).astype(np.complex64)
    M, Mo = build_M(pwa, A, 1.5 * n), oracle.norm_matrix(A, 1.5 * n)
    d = np.sqrt(np.diag(Mo).real)
    assert d[N // 2] > 0
    assert np.max(np.abs(M - Mo) / np.outer(d, d)) <= 1e-12


@pytest.mark.parametrize("N", [21, 33, 40, 48])
def test_fp64_kernel_many_waves(pwa, N):  # noqa: F811
    """The FP64 kernel beyond 20 waves, which serves what the digits cannot."""
    A = sample(N, 20_001, 7)
    M, Mo = build_M(pwa, A, 30_000.0, kernel="fp64"), oracle.norm_matrix(A, 30_000.0)
    d = np.sqrt(np.diag(Mo).real)
    assert np.max(np.abs(M - Mo) / np.outer(d, d)) <= 1e-12
