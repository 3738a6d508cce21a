"""The pool of device and pinned memory against a CUDA runtime of the test's own, on the
host: pwa_pool.cu is compiled unchanged and linked with allocation functions that count,
fail on demand and check that the pool's lock is free while they run."""
import os
import subprocess

import pytest

from paper_1108_5673_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1108_5673_gb300", "csrc")

RUNTIME = r'''
#include <stdio.h>
#include <stdlib.h>
#include <atomic>
#include <functional>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
#include <cuda_runtime.h>
#include <cuda.h>

namespace pwa {
cudaError_t pool_alloc(void **p, size_t bytes);
void pool_free(void *p, bool keep);
cudaError_t pool_host_alloc(void **p, size_t bytes);
void pool_host_free(void *p, bool keep);
size_t pool_trim();
void pool_loaded();
}

static std::mutex m;
static std::map<void *, size_t> dev, host;
static size_t limit = (size_t)1 << 40, dev_bytes = 0;
static const size_t kTotal = (size_t)32 << 30;   // so that 1 GB may be kept
static std::atomic<int> frees{0};
static std::atomic<bool> hook_on{false};
static std::function<void()> hook;
static thread_local int current = 0;
static unsigned long long context_id[2] = {11, 12};

static void run_hook()
{
    bool on = true;
    if (hook_on.compare_exchange_strong(on, false))
        hook();
}
static cudaError_t get(std::map<void *, size_t> &t, void **p, size_t n, size_t lim)
{
    run_hook();
    std::lock_guard<std::mutex> g(m);
    if (&t == &dev && dev_bytes + n > lim)
        return cudaErrorMemoryAllocation;
    *p = malloc(16);
    t[*p] = n;
    if (&t == &dev)
        dev_bytes += n;
    return cudaSuccess;
}
static cudaError_t put(std::map<void *, size_t> &t, void *p)
{
    if (!p)
        return cudaSuccess;
    run_hook();
    std::lock_guard<std::mutex> g(m);
    auto it = t.find(p);
    if (it == t.end())
        return cudaErrorInvalidValue;
    if (&t == &dev)
        dev_bytes -= it->second;
    t.erase(it);
    free(p);
    ++frees;
    return cudaSuccess;
}
extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return get(dev, p, n, limit); }
cudaError_t cudaFree(void *p) { return put(dev, p); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return get(host, p, n, limit); }
cudaError_t cudaFreeHost(void *p) { return put(host, p); }
cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *t = kTotal; *f = kTotal; return cudaSuccess; }
static CUresult ctx_id(CUcontext, unsigned long long *id) { *id = context_id[current]; return CUDA_SUCCESS; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *f = (void *)ctx_id;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); exit(1); } } while (0)
using namespace pwa;
static const size_t MB = (size_t)1 << 20;
static void *take(size_t n, bool h = false)
{
    void *p = nullptr;
    CHECK((h ? pool_host_alloc(&p, n) : pool_alloc(&p, n)) == cudaSuccess);
    return p;
}

int main()
{
    // a block is kept and taken again; one that must not be kept, or is too large, is not
    void *a = take(100 * MB);
    pool_free(a, true);
    CHECK(take(100 * MB) == a && frees == 0);
    pool_free(a, false);
    CHECK(frees == 1);
    pool_free(take(1025 * MB), true);
    CHECK(frees == 2 && dev.empty());
    // at most 1/32: the oldest go
    std::vector<void *> v;
    for (int i = 0; i < 12; ++i)
        v.push_back(take(100 * MB));
    for (void *p : v)
        pool_free(p, true);
    CHECK(dev.size() == 10 && dev_bytes <= kTotal / 32);
    // device and pinned blocks that eight loads did not take are freed at the ninth
    pool_host_free(take(MB, true), true);
    CHECK(host.size() == 1);
    for (int i = 0; i < 8; ++i)
        pool_loaded();
    CHECK(dev.size() == 10 && host.size() == 1);
    pool_loaded();
    CHECK(dev.empty() && host.empty());
    // trim gives back both kinds and says how much; blocks in use stay
    void *used = take(10 * MB);
    pool_free(take(20 * MB), true);
    pool_host_free(take(2 * MB, true), true);
    CHECK(pool_trim() == 22 * MB && dev.size() == 1 && host.empty());
    CHECK(pool_trim() == 0);
    // a failed allocation frees what is kept and is tried again; with nothing kept it fails
    pool_free(take(500 * MB), true);
    limit = 600 * MB;
    void *b = take(550 * MB);
    CHECK(dev.size() == 2);
    void *none;
    CHECK(pool_alloc(&none, 600 * MB) == cudaErrorMemoryAllocation && !none);
    limit = (size_t)1 << 40;
    pool_free(b, true);
    pool_free(used, true);
    CHECK(pool_trim() == 560 * MB);
    // the lists of another device, and of a context that was reset, are its own
    pool_free(take(30 * MB), true);
    current = 1;
    CHECK(pool_trim() == 0);
    current = 0;
    context_id[0] = 21;
    CHECK(pool_trim() == 0);
    // CUDA's own calls run without the pool's lock: another thread gets through meanwhile
    for (int kind = 0; kind < 4; ++kind) {
        bool through = false;
        hook = [&] {
            std::thread t([&] {
                void *p = nullptr;
                pool_alloc(&p, 4 * MB);
                pool_free(p, true);
                through = true;
            });
            t.join();
        };
        void *p = take(50 * MB);
        if (kind == 3)
            pool_free(take(40 * MB), true);
        hook_on = true;
        if (kind == 0)
            take(60 * MB);
        else if (kind == 1)
            pool_free(p, false);
        else if (kind == 2)
            take(3 * MB, true);
        else
            pool_trim();
        CHECK(through);
    }
    // several threads
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([t] {
            unsigned r = t + 1;
            std::vector<void *> mine;
            for (int i = 0; i < 20000; ++i) {
                r = r * 1664525u + 1013904223u;
                if (mine.size() < 6 && (r >> 20) % 2) {
                    mine.push_back(take(((r >> 8) % 64 + 1) * MB));
                } else if (!mine.empty()) {
                    pool_free(mine.back(), (r >> 12) % 8 != 0);
                    mine.pop_back();
                }
                if (r % 97 == 0)
                    pool_loaded();
                if (r % 193 == 0)
                    pool_trim();
            }
            for (void *p : mine)
                pool_free(p, true);
        });
    for (auto &t : ts)
        t.join();
    return 0;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("pool")
    (d / "t.cpp").write_text(RUNTIME)
    exe = d / "t"
    cmd = [build.nvcc(), "-std=c++17", "-O1", "-cudart", "none", "--expt-relaxed-constexpr"] + build.ARCH
    # registration stubs that nvcc's host code may refer to
    (d / "s.cpp").write_text('extern "C" { void **__cudaRegisterFatBinary(void *) { return nullptr; }\n'
                             'void __cudaRegisterFatBinaryEnd(void **) {}\n'
                             'void __cudaUnregisterFatBinary(void **) {}\n'
                             'char __cudaInitModule(void **) { return 0; } }\n')
    r = subprocess.run(cmd + ["-o", str(exe), str(d / "t.cpp"), str(d / "s.cpp"), os.path.join(CSRC, "pwa_pool.cu"),
                              "-Xcompiler", "-pthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return exe


@pytest.mark.timeout(120)
def test_pool(program):
    env = dict(os.environ)
    env.pop("PWA_POOL", None)
    r = subprocess.run([str(program)], capture_output=True, text=True, timeout=100, env=env)
    assert r.returncode == 0, r.stdout + r.stderr
