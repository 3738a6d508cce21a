"""The TMA-fed incoherent kernel at the edges of its units (64 events), tiles (three
units) and ring (up to 18 units), with one and with two gradient warps to a unit."""

import numpy as np
import pytest

import oracle
import synth
from test_gpu_incoh import case, check_sets, pwa  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L", [(4, 2), (7, 4), (12, 4), (20, 2), (23, 2)])
@pytest.mark.parametrize("units", [1, 3, 3 * 152, 3 * 152 * 7 + 1])
@pytest.mark.parametrize("off", [-1, 0, 1])
def test_edges(pwa, N, L, units, off):  # noqa: F811
    wl = case(N, L, 64 * units + off, 400, seed=units % 91 + off)
    Vs = [synth.random_V(N, 3 + units % 7), synth.random_V(N, 5)]
    with pwa.Likelihood(N, max_k=2) as lik:
        lik.load_events(wl.A_data, wl.A_mc, wl.n_gen)
        M = lik.build_norm()
        nll, g = lik.nll_grad(np.stack(Vs))
        again = lik.nll_grad(np.stack(Vs))
    assert np.array_equal(nll, again[0]) and np.array_equal(g, again[1])
    check_sets(nll, g, wl, M, Vs)
