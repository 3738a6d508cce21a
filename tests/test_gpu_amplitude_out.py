"""Generated amplitudes into any buffer the C entry points take: host memory, and
device memory at any multiple of a float (the kernels store whole complex numbers
where the buffer is aligned to them)."""
import ctypes

import numpy as np
import pytest

import synth
from test_gpu_norm import pwa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 1000])
@pytest.mark.parametrize("covariant", [False, True])
def test_offset_by_a_float(pwa, covariant, n):  # noqa: F811
    import torch
    rng = np.random.default_rng(n)
    if covariant:
        waves = [(1.0 + 0.2 * k, 0.1, 2 * (k % 2)) for k in range(5)]
        x = rng.standard_normal((n, 9))
    else:
        waves = synth.waves_linear(7)
        ev = synth.phase_space(n, np.random.Generator(np.random.Philox(n)))
        x = np.ascontiguousarray(np.stack([ev["m"], ev["costh"], ev["phi"]], axis=1))
    name = "pwa_compute_covariant_amplitudes" if covariant else "pwa_compute_amplitudes"
    size = 2 * n * len(waves) * (4 if covariant else 1)
    from paper_1108_5673_gb300 import _abi
    with pwa.Likelihood(len(waves)) as L:
        want = (L.covariant_amplitudes if covariant else L.amplitudes)(waves, x).view(np.float32).ravel()
        for offset in (0, 1, 2, 3):
            buf = torch.full((size + 8,), -7.0, device="cuda")
            table = (_abi._cov_waves if covariant else _abi._waves)(waves)
            assert getattr(_abi.load(), name)(L.ctx, table, x.ctypes.data_as(ctypes.c_void_p), n,
                                              ctypes.c_void_p(buf.data_ptr() + 4 * offset)) == 0
            got = buf.cpu().numpy()
            assert np.array_equal(got[offset:offset + size].view(np.int32), want.view(np.int32))
            assert np.all(got[:offset] == -7) and np.all(got[offset + size:] == -7)
