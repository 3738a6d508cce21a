"""M is the same bits on every run: nothing in the tensor-core kernel may read a
stage, a digit buffer or an accumulator while it is being refilled. A stage is
released once its amplitudes are in registers, and refilled within a microsecond;
a warp that had not read them yet would take single rows from the next tile (an
error of one tile's share, ~1e-4, in one wave's entries, in some runs)."""
import numpy as np
import pytest
import torch

from test_gpu_norm import pwa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(4, 300_000), (12, 300_000), (20, 300_000), (24, 200_000),
                                 (28, 400_000), (32, 1_000_000), (41, 200_000), (48, 400_000)])
def test_same_bits(pwa, N, n):  # noqa: F811
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    A = torch.view_as_complex(torch.randn(n, N, 2, generator=g, device="cuda"))
    with pwa.Likelihood(N) as L:
        L.load_events(A[:1].contiguous(), A, 2.0 * n)
        first = L.build_norm()
        for _ in range(60):
            assert np.array_equal(first, L.build_norm())
    X = torch.view_as_real(A).reshape(n, -1).double()
    G = (X.T @ X).cpu().numpy() / (2.0 * n)
    M = G[0::2, 0::2] + G[1::2, 1::2] + 1j * (G[0::2, 1::2] - G[1::2, 0::2])
    d = np.sqrt(np.diag(M).real)
    assert np.max(np.abs(first - M) / np.outer(d, d)) <= 1e-12
