"""Memory kept between contexts: results do not depend on what a block held
before, contexts may come and go in several threads, and kept memory is
bounded and given back (a block that eight sample loads did not take is freed;
at most 1/32 of the device is kept; PWA_POOL=0 keeps nothing)."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def pwa():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1108_5673_gb300 as pkg
    return pkg


def session(pwa, wl, V, forms, K):
    with pwa.Likelihood(len(V[0]), forms=forms, max_k=K) as L:
        L.load_events(wl.A_data, wl.A_mc, wl.n_gen)
        out = [L.build_norm()]
        for form in (pwa.PWA_FORM_AMP, pwa.PWA_FORM_TABLE, pwa.PWA_FORM_TC):
            if forms & form:
                L.set_form(form)
                out += list(L.nll_grad(V))
        return out + [L.hessian(V[0]), L.mc_weights(V[0])]


def samples(pwa):
    every = pwa.PWA_FORM_AMP | pwa.PWA_FORM_TABLE | pwa.PWA_FORM_TC
    out = []
    for N, n, forms in ((5, 3001, every), (20, 40_000, every), (33, 9_999, pwa.PWA_FORM_AMP), (20, 777, every)):
        wl = synth.mixture_workload("p", synth.waves_linear(N), n, 2 * n + 1, seed_data=N, seed_mc=n)
        out.append((wl, synth.random_V(N, 3, 3), forms))
    return out


def same(a, b):
    return len(a) == len(b) and all(np.array_equal(x, y) for x, y in zip(a, b))


def test_results_do_not_depend_on_reused_memory(pwa):
    cases = samples(pwa)
    first = [session(pwa, wl, V, f, 3) for wl, V, f in cases]
    for _ in range(3):
        for k in (1, 0, 3, 2, 1):
            wl, V, f = cases[k]
            assert same(first[k], session(pwa, wl, V, f, 3)), k


def test_contexts_in_threads(pwa):
    cases = samples(pwa)
    want = [session(pwa, wl, V, f, 3) for wl, V, f in cases]
    bad = []

    def work(k):
        wl, V, f = cases[k]
        for _ in range(5):
            try:
                if not same(want[k], session(pwa, wl, V, f, 3)):
                    bad.append(k)
            except pwa.PwaError as e:
                bad.append((k, str(e)))

    threads = [threading.Thread(target=work, args=(k % len(cases),)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad


CHILD = r'''
import sys
sys.path.insert(0, sys.argv[1])
import torch
import paper_1108_5673_gb300 as pwa

def load(n, N=20):
    A = torch.ones(n, N, dtype=torch.complex64, device="cuda")
    L = pwa.Likelihood(N)
    L.load_events(A[: n // 2], A, float(n))
    return L

load(1000).close()
torch.cuda.empty_cache()
torch.cuda.synchronize()
used = [torch.cuda.mem_get_info()[0]]
load(4_000_000).close()          # 960 MB of planes
torch.cuda.empty_cache()
used.append(torch.cuda.mem_get_info()[0])
for _ in range(10):
    load(1000).close()
torch.cuda.empty_cache()
used.append(torch.cuda.mem_get_info()[0])
print((used[0] - used[1]) >> 20, (used[0] - used[2]) >> 20)
'''


@pytest.mark.parametrize("pool", ["1", "0"])
def test_kept_memory_is_given_back(pwa, pool):
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=dict(os.environ, PWA_POOL=pool),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    after, later = map(int, r.stdout.split())
    if pool == "1":
        assert 900 <= after <= 1100, after
    else:
        assert after <= 64, after
    assert later <= 64, later
