"""M beyond 20 waves is as accurate as FP64 sums of exact products: what five
digits leave of an amplitude is multiplied too, rounded to 8 bits of its own.

Bound: with x the amplitude in units of 2^r and z = x minus its nearest multiple of
2^-40, an entry of G = X X^T misses sum_j x_p e_q + e_p x_q with |e| <= 2^-9 |z| of
random sign, standard deviation at most 2^-9 sqrt(sum_j x_p^2 z_q^2 + z_p^2 x_q^2);
M combines two such entries; six standard deviations, plus 1e-15 of sqrt(M_aa M_bb) for
the sums (FP64's own is 1.4e-15 on these samples). The reference adds exact products
in FP64 over 512 events at a time, the parts in extended precision.
"""
import numpy as np
import pytest

import synth
from test_gpu_norm import build_M, pwa  # noqa: F401

pytestmark = pytest.mark.gpu


def real_rows(A):
    A = A.astype(np.complex64)
    X = np.empty((A.shape[0], 2 * A.shape[1]), np.float64)
    X[:, 0::2], X[:, 1::2] = A.real, A.imag
    amax = (np.abs(A.real) + np.abs(A.imag)).max(axis=0).astype(np.float64)
    r = np.repeat(np.floor(np.log2(amax)) + 2, 2)
    return X, 2.0 ** r


def combine(G):
    return G[0::2, 0::2] + G[1::2, 1::2], G[0::2, 1::2] - G[1::2, 0::2]


def reference(X):
    G = np.zeros((X.shape[1],) * 2, np.longdouble)
    for i in range(0, X.shape[0], 512):
        x = X[i:i + 512]
        G += x.T @ x
    return combine(G)


@pytest.mark.parametrize("N,n_mc", [(21, 50_000), (24, 1_025), (28, 60_001), (32, 200_000), (33, 20_000),
                                    (40, 50_000), (48, 60_000)])
def test_error(pwa, N, n_mc):  # noqa: F811
    wl = synth.mixture_workload("n", synth.waves_linear(N), 10, n_mc, seed_mc=700 + N)
    X, s = real_rows(wl.A_mc)
    x = X / s
    z = x - np.rint(x * 2.0 ** 40) * 2.0 ** -40
    assert np.any(z != 0)
    re, im = reference(X)
    d = np.sqrt(np.diag(re))
    dd = np.outer(d, d).astype(np.float64)
    var = (x * x).T @ (z * z)
    sd = np.sqrt(var + var.T) * np.outer(s, s)
    sd = np.sqrt(sd[0::2, 0::2] ** 2 + sd[1::2, 1::2] ** 2 + sd[0::2, 1::2] ** 2 + sd[1::2, 0::2] ** 2)
    M = build_M(pwa, wl.A_mc, wl.n_gen)
    bound = 6 * 2.0 ** -9 * sd + 1e-15 * dd
    ng = np.longdouble(wl.n_gen)
    assert np.all(np.abs(M.real * ng - re) <= bound), np.max(np.abs(M.real * ng - re) / dd)
    assert np.all(np.abs(M.imag * ng - im) <= bound), np.max(np.abs(M.imag * ng - im) / dd)


@pytest.mark.parametrize("N", [21, 40])
def test_narrow_resonances(pwa, N):  # noqa: F811
    """A wave whose largest amplitude is far above its rms (a resonance of 1e-4 GeV; one
    event of 2000 times the others' size) keeps the FP64 kernel's accuracy: M is that
    kernel's. (Without M asked for too: the fit fractions are those of its M.)"""
    rng = np.random.default_rng(N)
    n = 20_000
    A = (rng.standard_normal((n, N)) + 1j * rng.standard_normal((n, N))).astype(np.complex64)
    m = rng.uniform(0.98, 3.0, n)
    B, C = A.copy(), A.copy()
    B[:, 3] = (1 / (1.5 ** 2 - m * m - 1j * 1.5 * 1e-4)).astype(np.complex64)
    C[5, 7] = 2000
    for S in (B, C):
        assert np.array_equal(build_M(pwa, S, 1.5 * n), build_M(pwa, S, 1.5 * n, kernel="fp64"))
    assert not np.array_equal(build_M(pwa, A, 1.5 * n), build_M(pwa, A, 1.5 * n, kernel="fp64"))
    V = np.ones(N, complex)
    with pwa.Likelihood(N) as L:
        L.load_events(B[:10], B, 1.5 * n)
        M = L.build_norm()
        F = L.fit_fractions(V)
        L.load_events(B[:10], B, 1.5 * n)
        assert L._abi.load().pwa_build_norm(L.ctx, None) == 0
        assert np.array_equal(F, L.fit_fractions(V))
