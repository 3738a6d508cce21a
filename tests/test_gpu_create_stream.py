"""A context's scratch is cleared before the context uses it, whatever else is queued
on the device: with kept memory nothing between pwa_create and the first evaluation
waits for the default stream. (M by the FP64 kernel and not copied out, so that no
blocking copy waits either.)"""
import os

import numpy as np
import pytest

import synth
from test_gpu_norm import pwa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture
def fp64_norm():
    os.environ["PWA_NORM_KERNEL"] = "fp64"
    yield
    del os.environ["PWA_NORM_KERNEL"]


def test_default_stream_busy(pwa, fp64_norm):  # noqa: F811
    import torch
    wl = synth.mixture_workload("s", synth.waves_linear(20), 5000, 3000, seed_data=1, seed_mc=2)
    V = synth.random_V(20, 4, 3)

    def session():
        with pwa.Likelihood(20, max_k=3) as L:
            L.load_events(wl.A_data, wl.A_mc, wl.n_gen)
            assert L._abi.load().pwa_build_norm(L.ctx, None) == 0
            return [L.nll_grad(V) for _ in range(50)]

    pwa.trim()      # no block left by others to be freed, which would wait, meanwhile
    want = session()[0]
    session()
    for _ in range(3):
        busy = torch.cuda.Event()
        torch.cuda._sleep(400_000_000)      # 0.2 s on the default stream
        busy.record()
        got = session()
        waited = busy.query()
        for nll, g in got:
            assert np.array_equal(nll, want[0]) and np.array_equal(g, want[1])
        torch.cuda.synchronize()
        assert not waited, "the session itself waited for the default stream: nothing was tested"

