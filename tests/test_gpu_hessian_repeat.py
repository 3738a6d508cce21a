"""The tensor-core Hessian is the same bits on every run: no stage is refilled while a
warp still reads it (see test_gpu_norm_repeat)."""
import numpy as np
import pytest
import torch

from test_gpu_norm import pwa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,n", [(4, 1_000_000), (12, 600_000), (19, 400_000), (20, 1_000_000)])
def test_same_bits(pwa, N, n):  # noqa: F811
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    A = torch.view_as_complex(torch.randn(n, N, 2, generator=g, device="cuda"))
    V = np.random.default_rng(N).standard_normal(N) + 1j
    with pwa.Likelihood(N) as L:
        L.load_events(A, A[:1000].contiguous(), 2000.0)
        first = L.hessian(V)
        for _ in range(200):
            assert np.array_equal(first, L.hessian(V))
    S = A.to(torch.complex128) @ torch.tensor(V, device="cuda")
    d = 2 * A.conj().to(torch.complex128) * (S / (S * S.conj()).real)[:, None]
    J = torch.cat([d.real, d.imag], dim=1)
    H = (J.T @ J).cpu().numpy()
    s = np.sqrt(np.diag(H))
    assert np.max(np.abs(first - H) / np.outer(s, s)) <= 1e-4
