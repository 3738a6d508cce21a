"""The tensor-core form's protocol for up to 16 parameter sets (k_batched.cu with two
accumulator buffers), under random schedules on the CPU: one step per tile, even
tiles to the first eight epilogue warps and buffer, odd ones to the others; R' is
shared. Same model and rules as test_batched_protocol_cpu.py."""
import random

import pytest

from test_batched_protocol_cpu import Bar

W = 8   # warps of a group


def simulate(n_tiles, NXS, seed, lag_rule=True, waits_r_free=True):
    rnd = random.Random(seed)
    x_full, x_empty = [Bar(1) for _ in range(NXS)], [Bar(1) for _ in range(NXS)]
    s_full, s_free = [Bar(1), Bar(1)], [Bar(W), Bar(W)]
    r_full, r_free, g_done = Bar(W), Bar(1), Bar(1)
    ops, S, read, rows, g2_done, x = [], [None, None], {}, {}, set(), {}

    def retire():
        kind, arg = ops.pop(0)
        if kind == "g1":
            assert arg < 2 or read.get(arg - 2, 0) == W, "S overwritten before it was read"
            S[arg & 1] = arg
        elif kind == "g2":
            assert x.get(arg % NXS) == arg, "X stage refilled before GEMM 2 read it"
            g2_done.add(arg)
        else:
            arg.arrive()

    def producer():
        for j in range(n_tiles):
            u = j // NXS
            while u > 0 and not x_empty[j % NXS].passes((u & 1) ^ 1):
                yield
            x[j % NXS] = j
            x_full[j % NXS].arrive()
            yield

    def issuer():
        g2 = ready = 0
        for q in range(n_tiles + 1):
            last = q == n_tiles
            need = ready if last else (q - 1 if lag_rule else 0)
            wx, ws = not last, not last and q >= 2
            while True:
                if g2 < ready and r_full.passes(g2 & 1):
                    assert rows.get(g2, 0) == W, "GEMM 2 on an incomplete R'"
                    ops.extend([("g2", g2), ("commit", r_free), ("commit", x_empty[g2 % NXS])])
                    g2 += 1
                    yield
                    continue
                if g2 >= need:
                    wx = wx and not x_full[q % NXS].passes((q // NXS) & 1)
                    ws = ws and not s_free[q & 1].passes((q // 2 - 1) & 1)
                    if not wx and not ws:
                        break
                yield
            if not last:
                assert x.get(q % NXS) == q
                ops.extend([("g1", q), ("commit", s_full[q & 1])])
                ready = q + 1
            yield
        ops.append(("commit", g_done))

    def warp(grp):
        for q in range(grp, n_tiles, 2):
            while not s_full[grp].passes((q // 2) & 1):
                yield
            assert S[grp] == q, "S does not hold this step"
            yield
            read[q] = read.get(q, 0) + 1
            s_free[grp].arrive()
            for _ in range(rnd.randint(0, 6)):
                yield
            if waits_r_free and q >= 1:
                while not r_free.passes((q - 1) & 1):
                    yield
            assert q == 0 or q - 1 in g2_done, "R' overwritten before GEMM 2 finished"
            rows[q] = rows.get(q, 0) + 1
            r_full.arrive()
            yield

    alive = [producer(), issuer()] + [warp(g) for g in (0, 1) for _ in range(W)]
    for _ in range(1_000_000):
        if not alive and not ops:
            break
        if ops and (not alive or rnd.random() < 0.3):
            retire()
            continue
        a = rnd.choice(alive)
        try:
            next(a)
        except StopIteration:
            alive.remove(a)
    else:
        raise RuntimeError("deadlock")
    assert g_done.C == 1


@pytest.mark.parametrize("n_tiles", [0, 1, 2, 3, 8, 17])
@pytest.mark.parametrize("NXS", [2, 3, 6])
def test_no_hazard(n_tiles, NXS):
    for seed in range(40):
        simulate(n_tiles, NXS, seed)


@pytest.mark.parametrize("rule", ["lag_rule", "waits_r_free"])
def test_each_rule_is_needed(rule):
    """Planted mistakes: without either rule some schedule overwrites R' too early."""
    failed = 0
    for seed in range(200):
        try:
            simulate(12, 3, seed, **{rule: False})
        except AssertionError:
            failed += 1
    assert failed
