"""The float-float amplitude generator against its FP64 evaluation
(PWA_AMPGEN_KERNEL=fp64): both give the float nearest to the model's value, so
they agree bitwise except where FP64's own rounding (2^-49 of the amplitude)
straddles a rounding boundary of float, less than one component in 10^6; there
they differ by one unit in the last place.
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


def both(pwa, waves, kin):
    with pwa.Likelihood(len(waves)) as L:
        A = L.amplitudes(waves, kin)
        os.environ["PWA_AMPGEN_KERNEL"] = "fp64"
        try:
            return A.view(np.float32), L.amplitudes(waves, kin).view(np.float32)
        finally:
            del os.environ["PWA_AMPGEN_KERNEL"]


def agree(a, b):
    d = a.view(np.int32) != b.view(np.int32)
    d &= ~(np.isnan(a) & np.isnan(b))
    x, y = a[d].astype(np.float64), b[d].astype(np.float64)
    assert np.all(np.abs(x - y) <= np.spacing(np.abs(b[d])))
    assert d.sum() <= max(2, 1e-6 * a.size), d.sum()


def kinematics(n, seed):
    ev = synth.phase_space(n, np.random.Generator(np.random.Philox(seed)))
    return np.stack([ev["m"], ev["costh"], ev["phi"]], axis=1)


LISTS = {
    "benchmark": synth.waves_linear(20),
    "one": synth.waves_linear(1),
    "largest": synth.waves_linear(48),
    "high l": [(1.0 + 0.04 * k, 0.05 + 0.01 * (k % 7), l, m) for k, (l, m) in enumerate(
        (l, m) for l in (16, 9, 3, 12, 1, 0, 7) for m in (l, -l, 0, -(l // 2), l // 3, -1 if l else 0))],
    "narrow": [(1.019461, 0.004249, 1, 1), (3.0969, 9.3e-5, 1, -1), (1.5, 1e-9, 2, 0), (0.1, 10.0, 4, -3)],
    "MeV": [(1500.0 + 100 * k, 100.0, k % 5, -(k % 3) if k % 5 >= k % 3 else 0) for k in range(7)],
    "outside": [(1e20, 1e15, 2, 1), (1.5, 1e-30, 0, 0)],
}


@pytest.mark.parametrize("name", LISTS)
@pytest.mark.parametrize("n", [1, 33, 100_003])
def test_wave_lists(pwa, name, n):
    kin = kinematics(n, 11 + n)
    if name == "MeV":
        kin[:, 0] *= 1000
    agree(*both(pwa, LISTS[name], kin))


def test_special_events(pwa):
    """Poles, axes, exact angles, angles of many turns, masses on resonance and
    zero, and values that are not numbers."""
    c = [-1.0, 1.0, 0.0, -0.0, 0.5, 1 - 2.0 ** -53, -1 + 2.0 ** -40, 1e-20, 1e-300, 1.5, np.nan]
    p = [0.0, -0.0, np.pi / 2, np.pi, -np.pi, 2 * np.pi, 1e-9, 1e-30, 1e5, -3e6, 1e15, np.inf]
    m = [0.0, 1.0, 1.1, 2.9, 1e-30, 1e30, np.inf, 0.98]
    kin = np.array([(x, y, z) for x in m for y in c for z in p])
    with np.errstate(all="ignore"):
        for waves in (LISTS["benchmark"], LISTS["high l"]):
            agree(*both(pwa, waves, kin))


def test_planes_equal_event_major(pwa):
    """The planes of a loaded sample hold the same floats: M of a generated
    sample equals M of the same amplitudes loaded as arrays, bitwise."""
    waves, kin = LISTS["high l"][:30], kinematics(20_011, 5)
    with pwa.Likelihood(30) as L:
        A = L.amplitudes(waves, kin)
        L.load_generated(waves, kin[:777], kin, 40_000.0)
        M = L.build_norm()
        L.load_events(A[:777], A, 40_000.0)
        assert np.array_equal(M, L.build_norm())
