"""The Hessian kernel of more than 20 waves over many tiles per block: more than
8 and more than 16 of the 256-event tiles, so that the FP32 sums are handed to
the long sums none, one and two times, at every layout of its product threads."""

import numpy as np
import pytest

import oracle
import synth
from test_gpu_fit_extras import H_TOL, case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pwa():
    import paper_1108_5673_gb300 as m
    return m


@pytest.mark.parametrize("N", [21, 24, 29, 32, 37, 45, 48])
@pytest.mark.parametrize("tiles", [3, 9, 17])
def test_runs_of_tiles(pwa, N, tiles):
    """A block of 5003 events repeated: the sum is known from the block's."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wl = case(N, 5003, 700, seed=N + tiles)
    copies, rest = divmod((tiles - 1) * sms * 256 + 77, 5003)
    A = np.concatenate([wl.A_data] * copies + [wl.A_data[:rest]])
    V = synth.random_V(N, N)
    whole, bad = oracle.hessian(wl.A_data, V)
    part, bad2 = oracle.hessian(wl.A_data[:rest], V)
    assert bad == 0 and bad2 == 0
    want = copies * whole + part
    with pwa.Likelihood(N) as L:
        L.load_events(A, wl.A_mc, wl.n_gen)
        L.build_norm()
        H = L.hessian(V)
        assert np.array_equal(H, H.T)
        assert np.max(np.abs(H - want)) <= H_TOL * np.max(np.abs(want))
        small = L.hessian(V * 2.0 ** 40) * 2.0 ** 80
        assert np.max(np.abs(small - want)) <= H_TOL * np.max(np.abs(want))
