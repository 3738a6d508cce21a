"""The time limit of the tensor-core form's issuer, which polls its barriers
without sleeping and serves products of the other GEMM in between: it must not run
out on a loop that is making progress, whichever of its polls did some work, and
must run out on one that waits for ever. The rule (poll_limit.cuh) is plain C++;
the loop here is the issuer's: a poll that serves goes straight to the next one."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1108_5673_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include <initializer_list>
#include "poll_limit.cuh"

// Polls until poll `done` (0: never); poll `served` and every `every`-th do some work
// instead of the check. Returns the poll at which the limit ran out, 0 if never.
static unsigned long run(unsigned long done, unsigned long served, unsigned long every, unsigned long most)
{
    const unsigned long long start = 1700000000000000000ull, limit = 2000000000ull, per_poll = 100;
    pwa::PollLimit wait;
    for (unsigned long it = 1; it <= most; ++it) {
        if (it == served || (every && it % every == 0))
            continue;
        if (it == done)
            return 0;
        if (wait.due() && wait.expired(start + it * per_poll, limit))
            return it;
    }
    return most;
}

int main()
{
    int bad = 0;
    for (unsigned long served = 1; served <= 1100; ++served)       // one poll that serves
        if (unsigned long at = run(5000, served, 0, 6000))
            printf("poll %lu serves: ran out at %lu\n", served, at), bad = 1;
    for (unsigned long every : {2ul, 3ul, 64ul, 128ul, 256ul, 257ul})
        if (unsigned long at = run(100001, 0, every, 200000))
            printf("every %lu-th serves: ran out at %lu\n", every, at), bad = 1;
    // a wait that never ends: 2 s of polls of 100 ns, then the next check
    const unsigned long at = run(0, 256, 0, 30000000);
    if (at < 20000000 || at > 20000000 + 1024)
        printf("an endless wait ran out at %lu\n", at), bad = 1;
    return bad;
}
'''


def test_limit(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[:2000]


def test_the_issuer_uses_it():
    src = open(os.path.join(CSRC, "k_batched.cu")).read()
    assert "limit.due()" in src and "limit.expired(" in src
