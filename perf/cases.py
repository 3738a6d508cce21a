"""Performance cases of the likelihood library: what a fitter has it do.

Each kind of case is one call (or the short sequence of calls) of the public
Python API that a fit program makes, on samples of the sizes that the
repository's benchmark, generator and tests use, and ragged sizes between:

  grad        one evaluation NLL + gradient, direct form, host call: the inner
              loop of every fit
  multistart  many starting points per call on the tensor cores
  free        one evaluation with free masses and widths
  models      one evaluation of several trial models, many starting points each
  hessian     FUMILI's Hessian, once per FUMILI step
  incoherent  one evaluation of a sample summed over unobserved components
  sample      a new sample: load, normalisation matrix, first evaluation
  generate    amplitudes BW x Y_l^m from kinematics, into a device buffer
  covariant   a new sample from 3-momenta: covariant amplitudes, load,
              normalisation matrix, first evaluation

Inputs follow the repository's synthetic samples: accepted Monte Carlo uniform
in (m, phi) with efficiency 0.6 + 0.3 cos(theta), data from a mixture of the
resonances, V normally distributed.
"""
import math
import random

import numpy as np
import torch

import paper_1108_5673_gb300 as pwa

M_LO, M_HI = 0.98, 3.0          # m(KK) range, GeV
M_PSI, M_K = 3.0969, 0.493677   # J/psi and kaon masses, GeV
EFF_MEAN = 0.6                  # mean of the efficiency 0.6 + 0.3 cos(theta)
CHUNK = 1 << 18                 # events per step of the 64-bit evaluations
MAX_INCOHERENT_WAVES = {2: 24, 3: 16, 4: 12}


def listed():
    return [
        # the small four-wave fit: launch and host latency
        {"name": "grad_10k_4", "kind": "grad", "waves": 4, "events": 10_000},
        # the paper-scale single fit, the benchmark's headline
        {"name": "grad_1M_20", "kind": "grad", "waves": 20, "events": 1_000_000},
        # the multistart sample of the benchmark, 256 starts per call
        {"name": "multistart_4M_32_k256", "kind": "multistart", "waves": 32, "events": 4_000_000,
         "sets": 256, "precision": "bfp16"},
        # the benchmark's free-resonance fit: 4 of 20 Breit-Wigners free
        {"name": "free_2M_20_r4", "kind": "free", "waves": 20, "free": 4, "events": 2_000_000,
         "mc": 5_000_000},
        # a scan of trial models with 8..48 waves, 16 starts each
        {"name": "models_16_k16", "kind": "models", "models": 16, "sets": 16, "sizes": 1108,
         "most_events": 1_000_000},
        # FUMILI's Hessian at the paper scale
        {"name": "hessian_1M_20", "kind": "hessian", "waves": 20, "events": 1_000_000},
        # and for a larger model on an odd-sized sample
        {"name": "hessian_333k_29", "kind": "hessian", "waves": 29, "events": 333_333},
        # two unobserved helicities per event
        {"name": "incoherent_1M_20_l2", "kind": "incoherent", "waves": 20, "components": 2,
         "events": 1_000_000, "mc": 2_000_000},
        # setting up the paper-scale sample and the multistart sample
        {"name": "sample_1M_5M_20", "kind": "sample", "waves": 20, "events": 1_000_000,
         "mc": 5_000_000, "dtype": "complex64"},
        {"name": "sample_4M_10M_32", "kind": "sample", "waves": 32, "events": 4_000_000,
         "mc": 10_000_000, "dtype": "complex64"},
        # the amplitudes of the paper-scale Monte Carlo sample
        {"name": "generate_5M_20", "kind": "generate", "waves": 20, "lmax": 4, "events": 5_000_000},
        # J/psi -> gamma K+ K- from momenta to the first evaluation
        {"name": "covariant_1M_12", "kind": "covariant", "waves": 12, "events": 1_000_000,
         "mc": 2_500_000},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["grad", "grad", "multistart", "free", "models", "hessian", "incoherent",
                       "sample", "generate", "covariant"])
    if kind == "grad":
        n = rng.randint(1, 48)
        return {"kind": kind, "waves": n, "events": log_int(1_000, min(4_000_000, 128_000_000 // n))}
    if kind == "multistart":
        n, k = rng.randint(4, 48), log_int(8, 256)
        most = min(4_000_000, 32 * 256 * 4_000_000 // (48 * k) if n > 32 else 4_000_000)
        return {"kind": kind, "waves": n, "events": log_int(50_000, most), "sets": k,
                "precision": rng.choice(["bfp16", "bfp16", "bfp8"])}
    if kind == "free":
        n = rng.randint(4, 32)
        e = log_int(20_000, min(2_000_000, 40_000_000 // n))
        return {"kind": kind, "waves": n, "free": rng.randint(1, min(8, n)), "events": e,
                "mc": 5 * e // 2}
    if kind == "models":
        return {"kind": kind, "models": rng.randint(3, 16), "sets": log_int(4, 32),
                "sizes": rng.randint(1, 1 << 30), "most_events": log_int(200_000, 1_000_000)}
    if kind == "hessian":
        return {"kind": kind, "waves": rng.randint(2, 48), "events": log_int(10_000, 1_000_000)}
    if kind == "incoherent":
        c = rng.randint(2, 4)
        e = log_int(10_000, 1_000_000)
        return {"kind": kind, "waves": rng.randint(2, MAX_INCOHERENT_WAVES[c]), "components": c,
                "events": e, "mc": 2 * e}
    if kind == "sample":
        n = rng.randint(4, 48)
        e = log_int(20_000, min(4_000_000, 128_000_000 // n))
        return {"kind": kind, "waves": n, "events": e, "mc": 5 * e // 2,
                "dtype": rng.choice(["complex64", "complex64", "complex128"])}
    if kind == "generate":
        n = rng.randint(2, 48)
        return {"kind": kind, "waves": n, "lmax": rng.choice([4, 4, 6, 10]),
                "events": log_int(20_000, min(5_000_000, 100_000_000 // n))}
    e = log_int(20_000, 1_000_000)
    return {"kind": kind, "waves": rng.randint(2, 12), "events": e, "mc": 5 * e // 2}


# ---- events and amplitudes, in 64 bits ------------------------------------------

def waves_of(n, lmax=4):
    """(mass, width, l, m) of n waves, masses and widths spread linearly. l
    cycles through 0, 2, 4 with m >= 0 (the benchmark's waves); for a larger
    lmax through 0..lmax with m of both signs."""
    out = []
    for a in range(n):
        t = a / (n - 1) if n > 1 else 0.0
        if lmax <= 4:
            l = (0, 2, 4)[a % 3]
            m = (a // 3) % (l + 1)
        else:
            l = a % (lmax + 1)
            m = (3 * a) % (2 * l + 1) - l
        out.append((1.0 + 1.9 * t, 0.05 + 0.35 * t, l, m))
    return out


def cov_waves_of(n):
    """(mass, width, spin) of n waves, spins 0 and 2 in turn."""
    return [(w[0], w[1], 2 * (a % 2)) for a, w in enumerate(waves_of(n))]


def rng_of(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000 + stream)
    return lambda n: torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def random_v(seed, waves, sets=None, scale=1.0):
    r = np.random.Generator(np.random.Philox(seed + 7))
    shape = (waves,) if sets is None else (sets, waves)
    return scale * (r.standard_normal(shape) + 1j * r.standard_normal(shape))


def accepted_cos(u):
    """cos(theta) with density 0.6 + 0.3 cos(theta) on [-1, 1], by inversion."""
    return (-0.6 + torch.sqrt(0.36 - 0.6 * (0.45 - 1.2 * u))) / 0.3


def mc_events(n, seed):
    """n accepted Monte Carlo events (m, cos theta, phi) and the number generated."""
    u = rng_of(seed, 1)
    return (M_LO + (M_HI - M_LO) * u(n), accepted_cos(u(n)), 2 * math.pi * u(n)), float(int(n / EFF_MEAN))


def data_events(n, waves, seed):
    """n data events, m from the Breit-Wigners of the waves in equal parts."""
    u = rng_of(seed, 2)
    mass = torch.tensor([w[0] for w in waves], device="cuda", dtype=torch.float64)
    half = torch.tensor([w[1] for w in waves], device="cuda", dtype=torch.float64) / 2
    a = torch.clamp((u(n) * len(waves)).long(), max=len(waves) - 1)
    mass, half = mass[a], half[a]
    lo = torch.atan((M_LO - mass) / half)
    hi = torch.atan((M_HI - mass) / half)
    m = torch.clamp(mass + half * torch.tan(lo + (hi - lo) * u(n)), M_LO, M_HI)
    return m, accepted_cos(u(n)), 2 * math.pi * u(n)


def legendre(l, m, x):
    """P_l^m(x), m >= 0, with the Condon-Shortley phase."""
    p = torch.ones_like(x)
    s = torch.sqrt(torch.clamp(1 - x * x, min=0.0))
    for k in range(m):
        p = p * (-(2 * k + 1)) * s
    if l == m:
        return p
    q = x * (2 * m + 1) * p
    for k in range(m + 2, l + 1):
        p, q = q, ((2 * k - 1) * x * q - (k + m - 1) * p) / (k - m)
    return q


def ylm(l, m, x, phi):
    k = abs(m)
    norm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - k) / math.factorial(l + k))
    y = torch.polar(norm * legendre(l, k, x), k * phi)
    if m < 0:
        y = (-1) ** k * y.conj()
    return y


def breit_wigner(m, mass, width):
    return 1.0 / torch.complex(mass * mass - m * m, torch.full_like(m, -mass * width))


def amplitudes(events, waves, dtype=torch.complex64, shift=0):
    """[n, waves] amplitudes; `shift` moves each m within -l..l (a helicity)."""
    m, x, phi = events
    out = torch.empty((m.shape[0], len(waves)), dtype=dtype, device="cuda")
    for a, (mass, width, l, k) in enumerate(waves):
        k = max(-l, min(l, k + shift))
        out[:, a] = breit_wigner(m, mass, width) * ylm(l, k, x, phi)
    return out


def radiative_momenta(n, seed, accepted):
    """[n, 9] 3-momenta (photon, K+, K-) of J/psi -> gamma X, X -> K+ K- in the
    J/psi rest frame, m(KK) and the directions uniform (`accepted`: the
    photon's cos theta with the efficiency)."""
    u = rng_of(seed, 3)
    m = 0.99 + (3.0 - 0.99) * u(n)
    cg = accepted_cos(u(n)) if accepted else 2 * u(n) - 1
    ck, pg, pk = 2 * u(n) - 1, 2 * math.pi * u(n), 2 * math.pi * u(n)
    sg, sk = torch.sqrt(1 - cg * cg), torch.sqrt(1 - ck * ck)
    eg = (M_PSI ** 2 - m * m) / (2 * M_PSI)
    q = eg[:, None] * torch.stack([sg * torch.cos(pg), sg * torch.sin(pg), cg], dim=1)
    ex = M_PSI - eg
    beta = -q / ex[:, None]
    b2 = (beta * beta).sum(1)
    gamma = ex / m
    k = torch.sqrt(m * m / 4 - M_K ** 2)
    ks = k[:, None] * torch.stack([sk * torch.cos(pk), sk * torch.sin(pk), ck], dim=1)
    bk = (beta * ks).sum(1)
    along = ((gamma - 1) * bk / b2)[:, None] * beta
    boost = (gamma * m / 2)[:, None] * beta
    return torch.cat([q, ks + along + boost, -ks - along + boost], dim=1)


def covariant_amplitudes(p3, waves):
    """[n, 4, waves] covariant tensor amplitudes (J/psi helicity +1, -1 times
    photon polarisation e1, e2) in 64 bits, as include/pwa.h states them."""
    n = p3.shape[0]
    zero = torch.zeros(n, device="cuda", dtype=torch.float64)
    q3, a3, b3 = p3[:, :3], p3[:, 3:6], p3[:, 6:]
    metric = torch.tensor([1.0, -1.0, -1.0, -1.0], device="cuda", dtype=torch.float64)

    def dot(a, b):
        return (a * b * metric).sum(-1)

    def four(v):
        return torch.cat([torch.sqrt(M_K ** 2 + (v * v).sum(1, keepdim=True)), v], dim=1)

    k1, k2 = four(a3), four(b3)
    p, r = k1 + k2, k1 - k2
    pp = dot(p, p)
    rt = r - (dot(r, p) / pp)[:, None] * p
    qh = q3 / torch.linalg.norm(q3, dim=1, keepdim=True)
    t = torch.sqrt(qh[:, 0] ** 2 + qh[:, 1] ** 2)
    e1 = torch.stack([zero, -qh[:, 1] / t, qh[:, 0] / t, zero], dim=1)
    e2 = torch.cat([zero[:, None], torch.linalg.cross(qh, e1[:, 1:], dim=1)], dim=1)
    q2, q0 = pp / 4 - M_K ** 2, 0.197327
    b2 = torch.sqrt(13 / (q2 * q2 + 3 * q2 * q0 ** 2 + 9 * q0 ** 4))
    out = torch.empty((n, 4, len(waves)), device="cuda", dtype=torch.complex128)
    for i, sign in enumerate((-1.0, 1.0)):
        psi = torch.tensor([0, sign, -1j, 0], device="cuda", dtype=torch.complex128) / math.sqrt(2)
        for j, e in enumerate((e1, e2)):
            s0 = dot(psi, e)
            s2 = b2 * (dot(psi, rt) * dot(e, rt) - dot(rt, rt) / 3 * (s0 - dot(psi, p) * dot(e, p) / pp))
            for a, (mass, width, spin) in enumerate(waves):
                bw = 1.0 / torch.complex(mass * mass - pp, torch.full_like(pp, -mass * width))
                out[:, 2 * i + j, a] = bw * (s2 if spin == 2 else s0)
    return out


# ---- states -----------------------------------------------------------------------

def coherent_sample(case, seed, dtype=torch.complex64):
    waves = waves_of(case["waves"])
    events, n_gen = mc_events(case.get("mc") or 2 * case["events"], seed)
    return amplitudes(data_events(case["events"], waves, seed), waves, dtype), amplitudes(events, waves, dtype), n_gen


def incoherent_sample(case, seed):
    waves = waves_of(case["waves"])
    data = data_events(case["events"], waves, seed)
    events, n_gen = mc_events(case["mc"], seed)
    shifts = (1, -1, 0, 2)[:case["components"]]
    return (torch.stack([amplitudes(data, waves, shift=h) for h in shifts], dim=1),
            torch.stack([amplitudes(events, waves, shift=h) for h in shifts], dim=1), n_gen)


class ResonanceSample:
    """The fields that Likelihood.load_resonance_events reads, and a start."""

    def __init__(self, case, seed):
        waves, r = waves_of(case["waves"]), case["free"]
        self.n_free = r
        mc, self.n_gen = mc_events(case["mc"], seed)
        data = data_events(case["events"], waves, seed)
        for name, (m, x, phi) in (("data", data), ("mc", mc)):
            m = m.float().double()   # the library holds m in 32 bits
            y = torch.stack([ylm(l, k, x, phi) for _, _, l, k in waves[:r]], dim=1)
            setattr(self, "m_" + name, m)
            setattr(self, "Y_" + name, y.to(torch.complex64))
            setattr(self, "Afix_" + name, amplitudes((m, x, phi), waves[r:]))
        self.mass = np.array([1.01 * w[0] for w in waves[:r]])
        self.width = np.array([0.95 * w[1] for w in waves[:r]])


def model_sizes(case):
    r = random.Random(case["sizes"])
    return [(r.randint(8, 48), r.randint(100_000, case["most_events"])) for _ in range(case["models"])]


def model_sample(size, seed, j):
    return coherent_sample({"waves": size[0], "events": size[1]}, seed * 100 + j)


def kinematics(case, seed):
    events, _ = mc_events(case["events"], seed)
    return torch.stack(events, dim=1).contiguous()


def prepare(case, seed):
    kind, n = case["kind"], case.get("waves")
    s = {"kind": kind, "waves": n}
    if kind in ("grad", "hessian"):
        data, mc, n_gen = coherent_sample(case, seed)
        L = pwa.Likelihood(n)
        L.load_events(data, mc, n_gen)
        L.build_norm()
        s.update(L=L, V=random_v(seed, n))
    elif kind == "multistart":
        data, mc, n_gen = coherent_sample(case, seed)
        prec = pwa.PWA_PREC_BFP8 if case["precision"] == "bfp8" else pwa.PWA_PREC_BFP16
        L = pwa.Likelihood(n, forms=pwa.PWA_FORM_TC, max_k=case["sets"], precision=prec)
        L.load_events(data, mc, n_gen)
        L.build_norm()
        s.update(L=L, V=random_v(seed, n, case["sets"], 2.0))
    elif kind == "free":
        sample = ResonanceSample(case, seed)
        L = pwa.Likelihood(n)
        L.load_resonance_events(sample)
        s.update(L=L, V=random_v(seed, n), mass=sample.mass, width=sample.width)
    elif kind == "models":
        sizes = model_sizes(case)
        B = pwa.ModelBatch([w for w, _ in sizes], case["sets"])
        for j, size in enumerate(sizes):
            data, mc, n_gen = model_sample(size, seed, j)
            B.load_model(j, data, mc, n_gen)
            del data, mc
        s.update(B=B, V=[random_v(seed * 100 + j, w, case["sets"], 2.0) for j, (w, _) in enumerate(sizes)])
    elif kind == "incoherent":
        data, mc, n_gen = incoherent_sample(case, seed)
        L = pwa.Likelihood(n)
        L.load_events(data, mc, n_gen)
        L.build_norm()
        s.update(L=L, V=random_v(seed, n))
    elif kind == "sample":
        data, mc, n_gen = coherent_sample(case, seed, getattr(torch, case["dtype"]))
        s.update(data=data, mc=mc, n_gen=n_gen, V=random_v(seed, n))
    elif kind == "generate":
        s.update(L=pwa.Likelihood(n), table=waves_of(n, case["lmax"]), kin=kinematics(case, seed),
                 out=torch.empty((case["events"], n), dtype=torch.complex64, device="cuda"))
    elif kind == "covariant":
        s.update(table=cov_waves_of(n), data=radiative_momenta(case["events"], seed, False),
                 mc=radiative_momenta(case["mc"], seed + 500_000_000, True),
                 n_gen=float(int(case["mc"] / EFF_MEAN)), V=random_v(seed, n))
    else:
        raise ValueError("unknown kind %r" % kind)
    return s


def run(s):
    kind = s["kind"]
    if kind in ("grad", "multistart", "incoherent"):
        nll, grad = s["L"].nll_grad(s["V"])
        return {"nll": nll, "grad": grad}
    if kind == "free":
        nll, gv, gm, gw = s["L"].nll_grad_res(s["V"], s["mass"], s["width"])
        return {"nll": nll, "grad": gv, "grad_mass": gm, "grad_width": gw}
    if kind == "models":
        nll, grads = s["B"].nll_grad(s["V"])
        return {"nll": nll, "grads": grads}
    if kind == "hessian":
        return {"hessian": s["L"].hessian(s["V"])}
    if kind == "generate":
        return {"amplitudes": s["L"].amplitudes(s["table"], s["kin"], s["out"])}
    with pwa.Likelihood(s["waves"]) as L:
        if kind == "sample":
            L.load_events(s["data"], s["mc"], s["n_gen"])
        else:
            L.load_covariant(s["table"], s["data"], s["mc"], s["n_gen"])
        M = L.build_norm()
        nll, grad = L.nll_grad(s["V"])
    return {"M": M, "nll": nll, "grad": grad}


def work(case):
    kind, n, e = case["kind"], case.get("waves"), case.get("events")
    if kind == "grad":
        return {"bytes": 8.0 * n * e, "flops": 16.0 * n * e}
    if kind == "multistart":
        return {"bytes": 8.0 * n * e, "flops": 16.0 * n * e * case["sets"]}
    if kind == "free":
        both = e + case["mc"]
        return {"bytes": 4.0 * (1 + 2 * n) * both, "flops": (16.0 * n + 40.0 * case["free"]) * both}
    if kind == "models":
        cells = sum(w * k for w, k in model_sizes(case))
        return {"bytes": 8.0 * cells, "flops": 16.0 * cells * case["sets"]}
    if kind == "hessian":
        # S, the gradient of ln I, and the upper triangle of its outer products
        return {"bytes": 8.0 * n * e, "flops": e * (16.0 * n + 2.0 * n * (2 * n + 1))}
    if kind == "incoherent":
        cells = n * case["components"] * e
        return {"bytes": 8.0 * cells, "flops": 16.0 * cells}
    if kind == "sample":
        # each amplitude in once and into the store once; M and one evaluation
        size = 16.0 if case["dtype"] == "complex128" else 8.0
        return {"bytes": (size + 8.0) * n * (e + case["mc"]),
                "flops": 4.0 * n * (n + 1) * case["mc"] + 16.0 * n * e}
    if kind == "generate":
        return {"bytes": (24.0 + 8.0 * n) * e, "flops": 25.0 * n * e}
    both = e + case["mc"]
    return {"bytes": (72.0 + 32.0 * n) * both,
            "flops": (357.0 + 33.0 * n) * both + 16.0 * n * (n + 1) * case["mc"] + 64.0 * n * e}


# ---- the same in 64 bits, plain torch ----------------------------------------------

def norm_exact(mc, n_gen):
    """M of [n, waves] amplitudes."""
    M = torch.zeros((mc.shape[1], mc.shape[1]), device="cuda", dtype=torch.complex128)
    for a in mc.split(CHUNK):
        a = a.to(torch.complex128)
        M += a.mH @ a
    return M / n_gen


def nll_exact(data, M, V):
    """nll [K], grad [K, waves] of [n, components, waves] amplitudes."""
    V = torch.from_numpy(np.atleast_2d(V)).cuda()
    nll = torch.zeros(V.shape[0], device="cuda", dtype=torch.float64)
    grad = torch.zeros_like(V)
    for a in data.split(CHUNK // data.shape[1]):
        a = a.to(torch.complex128)
        S = a @ V.T
        I = (S.real ** 2 + S.imag ** 2).sum(1)
        nll -= torch.log(I).sum(0)
        R = S / I[:, None, :]
        grad -= (a.reshape(-1, a.shape[2]).mH @ R.reshape(-1, V.shape[0])).T
    MV = V @ M.T
    nll += (V.conj() * MV).sum(1).real
    return nll.cpu().numpy(), (grad + MV).cpu().numpy()


def free_exact(case, seed):
    s = ResonanceSample(case, seed)
    r = s.n_free
    V = torch.from_numpy(random_v(seed, case["waves"])).cuda()
    nll = 0.0
    gv = torch.zeros_like(V)
    gm = torch.zeros(r, device="cuda", dtype=torch.float64)
    gw = torch.zeros_like(gm)
    M = torch.from_numpy(s.mass).cuda()
    G = torch.from_numpy(s.width).cuda()
    for name in ("data", "mc"):
        parts = [getattr(s, k + name).split(CHUNK) for k in ("m_", "Y_", "Afix_")]
        for m, y, fixed in zip(*parts):
            bw = 1.0 / torch.complex(M * M - (m * m)[:, None], (-M * G).expand(m.shape[0], r))
            y = y.to(torch.complex128)
            a = torch.cat([bw * y, fixed.to(torch.complex128)], dim=1)
            S = a @ V
            I = S.real ** 2 + S.imag ** 2
            w = -1.0 / I if name == "data" else torch.full_like(I, 1.0 / s.n_gen)
            nll += float((-torch.log(I) if name == "data" else w * I).sum())
            gv += a.mH @ (w * S)
            d = (w * S.conj())[:, None] * y * V[:r] * bw * bw
            gm += 2 * (-d * torch.complex(2 * M, -G)).real.sum(0)
            gw += 2 * (1j * d * M).real.sum(0)
    return {"nll": nll, "grad": gv.cpu().numpy(), "grad_mass": gm.cpu().numpy(),
            "grad_width": gw.cpu().numpy()}


def hessian_exact(data, V):
    V = torch.from_numpy(V).cuda()
    H = torch.zeros((2 * data.shape[1], 2 * data.shape[1]), device="cuda", dtype=torch.float64)
    for a in data.split(CHUNK):
        a = a.to(torch.complex128)
        S = a @ V
        g = 2 * a.conj() * (S / (S.real ** 2 + S.imag ** 2))[:, None]
        d = torch.cat([g.real, g.imag], dim=1)
        H += d.T @ d
    return H.cpu().numpy()


def exact(case, seed):
    kind, n = case["kind"], case.get("waves")
    if kind == "free":
        return free_exact(case, seed)
    if kind == "generate":
        kin = kinematics(case, seed)
        return {"amplitudes": amplitudes((kin[:, 0], kin[:, 1], kin[:, 2]), waves_of(n, case["lmax"]),
                                         torch.complex128)}
    if kind == "models":
        nll, grads = [], []
        for j, size in enumerate(model_sizes(case)):
            data, mc, n_gen = model_sample(size, seed, j)
            f, g = nll_exact(data[:, None, :], norm_exact(mc, n_gen),
                             random_v(seed * 100 + j, size[0], case["sets"], 2.0))
            nll.append(f)
            grads.append(g)
        return {"nll": np.stack(nll), "grads": grads}
    if kind == "covariant":
        waves = cov_waves_of(n)
        data = covariant_amplitudes(radiative_momenta(case["events"], seed, False), waves)
        mc = covariant_amplitudes(radiative_momenta(case["mc"], seed + 500_000_000, True), waves)
        n_gen = float(int(case["mc"] / EFF_MEAN))
    elif kind == "incoherent":
        data, mc, n_gen = incoherent_sample(case, seed)
    else:
        dtype = getattr(torch, case.get("dtype", "complex64"))
        data, mc, n_gen = coherent_sample(case, seed, dtype)
        data, mc = data[:, None, :], mc[:, None, :]
    if kind == "hessian":
        return {"hessian": hessian_exact(data[:, 0, :], random_v(seed, n))}
    M = norm_exact(mc.reshape(-1, n), n_gen)
    if kind == "multistart":
        V = random_v(seed, n, case["sets"], 2.0)
    else:
        V = random_v(seed, n)
    nll, grad = nll_exact(data, M, V)
    if kind in ("sample", "covariant"):
        return {"M": M.cpu().numpy(), "nll": nll, "grad": grad}
    return {"nll": nll, "grad": grad}
