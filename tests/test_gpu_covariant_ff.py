"""The float-float covariant generator against its FP64 evaluation
(PWA_AMPGEN_KERNEL=fp64). Both give the float nearest to the formalism's
value, so they agree bitwise except where FP64's own rounding straddles a
rounding boundary of float: 2^-49 of the amplitude for ordinary events, less
than one component in 10^5, and there by one unit in the last place. Near the
threshold, the beam axis and the pole of a wave FP64 loses more digits itself
(p.p from the momenta, the difference M^2 - p.p): there the bound is one unit
in the last place of |A| plus 1e-12 |A|, as for the oracle.
"""
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pwa():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1108_5673_gb300 as pkg
    return pkg


def both(pwa, waves, p3):
    with pwa.Likelihood(len(waves)) as L:
        A = L.covariant_amplitudes(waves, p3)
        os.environ["PWA_AMPGEN_KERNEL"] = "fp64"
        try:
            return A, L.covariant_amplitudes(waves, p3)
        finally:
            del os.environ["PWA_AMPGEN_KERNEL"]


@pytest.mark.parametrize("N,n", [(1, 1), (2, 33), (7, 63), (12, 65), (12, 100_003), (48, 4097)])
def test_ordinary_events(pwa, N, n):
    p3, _ = synth.radiative_events(n, np.random.default_rng(7 + n))
    A, B = both(pwa, synth.cov_waves(N), p3)
    a, b = A.view(np.float32), B.view(np.float32)
    d = a.view(np.int32) != b.view(np.int32)
    assert np.all(np.abs(a[d].astype(np.float64) - b[d]) <= np.spacing(np.abs(b[d])))
    assert d.sum() <= max(2, 1e-5 * a.size), d.sum()


def near(A, B):
    mag = np.abs(B.astype(np.complex128))
    tol = np.spacing(mag.astype(np.float32)).astype(np.float64) + 1e-12 * mag
    for part in (np.real, np.imag):
        a, b = part(A).astype(np.float64), part(B).astype(np.float64)
        fine = np.isfinite(b)
        assert np.array_equal(fine, np.isfinite(a))
        assert np.all(np.abs(a - b)[fine] <= tol[fine])


def test_edges(pwa):
    """Threshold, the beam axis and just off it, the end of the mass range,
    masses on a wave's pole, and waves narrow and out of range."""
    g = np.random.default_rng(3)
    n = 4000
    m = np.concatenate([0.987354 + 10.0 ** g.uniform(-9, -2, n), 3.0969 - 10.0 ** g.uniform(-6, -1, n),
                        np.full(n, 1.5), g.uniform(0.99, 3.0, n)])
    cg = np.concatenate([g.uniform(-1, 1, 2 * n), np.repeat([1.0, -1.0], n // 2),
                         1 - 10.0 ** g.uniform(-14, -3, n)])
    pg, ck, pk = g.uniform(0, 6.28, 4 * n), g.uniform(-1, 1, 4 * n), g.uniform(0, 6.28, 4 * n)
    p3 = synth.radiative_kinematics(m, cg, pg, ck, pk)
    for waves in (synth.cov_waves(6), [(1.5, 0.1, 2), (1.5, 1e-3, 0), (3.0, 1e-7, 2)],
                  [(1e12, 1.0, 0), (1.5, 0.1, 2)]):
        near(*both(pwa, waves, p3))


def test_inputs_that_are_no_decay(pwa):
    """Momenta that do not balance, zeros, tiny, huge and non-finite ones."""
    g = np.random.default_rng(4)
    p3 = g.standard_normal((3000, 9))
    p3[:500, 0:3] = 0
    p3[500:800, 0:2] = 0
    p3[800:1000, 3:9] *= 1e-12
    p3[1000:1100] *= 1e25
    p3[1100, 4] = np.nan
    p3[1101, 0] = np.inf
    with np.errstate(all="ignore"):
        near(*both(pwa, synth.cov_waves(4), p3))
