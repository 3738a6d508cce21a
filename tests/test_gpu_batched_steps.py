"""The tensor-core form around the change between steps of 16 sets (up to 16) and of
32: every feature count in steps of 32 (the sweep of test_gpu_batched.py has five
sets), set counts at the edges of a warp's eight, and few and many tiles per CTA."""

import pytest

import synth
from test_gpu_batched import PRECISIONS, case, check, prec, pwa  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", PRECISIONS)
@pytest.mark.parametrize("N", [4, 13, 24, 32, 40, 48])
def test_waves_in_steps_of_32(pwa, N, p):  # noqa: F811
    wl = case(N, 3000, 4000, seed=N)
    check(pwa, wl, [synth.random_V(N, 31 + N + j) for j in range(17)], prec(pwa, p), idx=[0, 8, 15, 16])


@pytest.mark.parametrize("K", [7, 8, 9, 15, 16, 17])
@pytest.mark.parametrize("n_data", [128, 129, 5 * 152 * 128 + 1])
def test_edges(pwa, K, n_data):  # noqa: F811
    wl = case(8, n_data, 700, seed=n_data % 89)
    check(pwa, wl, [synth.random_V(8, 7 + j) for j in range(K)], prec(pwa, "BFP16"), idx=[0, 6, K - 1])
