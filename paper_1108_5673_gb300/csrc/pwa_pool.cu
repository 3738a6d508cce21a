// Device and pinned host memory of the library's contexts.
//
// A context that is created, loaded, evaluated and destroyed (a scan over
// samples or models) spends more time in cudaMalloc, cudaFree and their host
// counterparts than in its kernels: at 1M + 5M events x 20 waves 0.97 ms to
// free the planes, 0.25 ms each to create and destroy the context, of 2.3 ms
// in all; at 4M + 10M x 32 waves 2.8 ms to free 3.6 GB, of 5.9 ms. Freed
// blocks are therefore kept for the next context, within bounds:
//  - at most 1/32 of the device's memory (64 MB of pinned memory) is kept; what
//    exceeds it is freed at once, oldest first;
//  - a block, device or pinned, that the last 8 sample loads on its device did
//    not take is freed at the next load;
//  - an allocation that fails frees everything kept and is tried again;
//  - PWA_POOL=0 keeps nothing.
//  - pwa_trim gives back everything kept.
// Blocks are put back only when the work that may use them has finished (the
// callers wait for it), so that any stream may use them next. The lists are guarded
// by one mutex, which is not held while CUDA allocates or frees (a free waits for the
// device). A device reset invalidates them: they belong to one CUDA context, whose id
// is compared at each use, and are dropped with it.
#include <stdlib.h>
#include <string.h>

#include <mutex>
#include <unordered_map>
#include <vector>

#include <cudaTypedefs.h>

#include "pwa_internal.cuh"

namespace pwa {

namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned kKeepLoads = 8;
constexpr size_t kHostCap = (size_t)64 << 20;

struct Block {
    void *p;
    size_t size;
    unsigned stamp;
};

struct Pool {
    unsigned long long context = 0;
    std::unordered_map<void *, size_t> live;
    std::vector<Block> kept;  // oldest first
    size_t kept_bytes = 0, cap = 0;
    unsigned loads = 0;
};

struct State {
    std::mutex lock;
    Pool dev[kMaxDevices], host[kMaxDevices];
};

// never destroyed: contexts may outlive static destructors
State &state()
{
    static State *s = new State;
    return *s;
}

bool enabled()
{
    static const bool on = [] {
        const char *v = getenv("PWA_POOL");
        return !(v && strcmp(v, "0") == 0);
    }();
    return on;
}

// Blocks that have left the lists, freed when this goes out of scope (after the lock).
struct Released {
    bool host;
    std::vector<Block> blocks;
    explicit Released(bool h) : host(h) {}
    ~Released()
    {
        for (const Block &b : blocks)
            if ((host ? cudaFreeHost(b.p) : cudaFree(b.p)) != cudaSuccess)
                cudaGetLastError();
    }
};

// Takes the first n kept blocks off the list.
void drop(Pool &p, size_t n, Released *out)
{
    for (size_t i = 0; i < n; ++i) {
        p.kept_bytes -= p.kept[i].size;
        out->blocks.push_back(p.kept[i]);
    }
    p.kept.erase(p.kept.begin(), p.kept.begin() + n);
}

// The pool of the current CUDA context; blocks of a context that is gone are
// forgotten (its memory went with it).
void renew(Pool &p, unsigned long long id)
{
    if (id && p.context != id) {
        p.kept.clear();
        p.live.clear();
        p.kept_bytes = 0;
        p.context = id;
    }
}

size_t rounded(size_t bytes)
{
    if (bytes >= (size_t)1 << 20)
        return (bytes + ((size_t)2 << 20) - 1) >> 21 << 21;
    size_t s = 512;
    while (s < bytes)
        s <<= 1;
    return s;
}

// The smallest kept block of [size, 1.25 size], or null.
void *take(Pool &p, size_t size)
{
    size_t best = p.kept.size();
    for (size_t i = 0; i < p.kept.size(); ++i)
        if (p.kept[i].size >= size && p.kept[i].size <= size + size / 4 &&
            (best == p.kept.size() || p.kept[i].size < p.kept[best].size))
            best = i;
    if (best == p.kept.size())
        return nullptr;
    const Block b = p.kept[best];
    p.kept.erase(p.kept.begin() + best);
    p.kept_bytes -= b.size;
    p.live[b.p] = b.size;
    return b.p;
}

void put(Pool &p, void *q, bool keep, Released *out)
{
    const auto it = p.live.find(q);
    Block b{q, 0, p.loads};
    const bool known = it != p.live.end();  // else of a context that was reset
    if (known) {
        b.size = it->second;
        p.live.erase(it);
    }
    if (!known || !keep || !enabled() || b.size > p.cap) {
        out->blocks.push_back(b);
        return;
    }
    p.kept.push_back(b);
    p.kept_bytes += b.size;
    size_t n = 0, bytes = p.kept_bytes;
    while (bytes > p.cap)
        bytes -= p.kept[n++].size;
    drop(p, n, out);
}

// Blocks that the last kKeepLoads loads did not take.
void age(Pool &p, Released *out)
{
    ++p.loads;
    size_t n = 0;  // stamps grow along the list
    while (n < p.kept.size() && p.loads - p.kept[n].stamp > kKeepLoads)
        ++n;
    drop(p, n, out);
}

// The current device and the id of its context (false: no device).
bool where(int *dev, unsigned long long *id)
{
    if (cudaGetDevice(dev) != cudaSuccess || *dev < 0 || *dev >= kMaxDevices) {
        cudaGetLastError();
        return false;
    }
    *id = cuda_context_id();
    return true;
}

// (with the lock held)
Pool &pool_of(int dev, unsigned long long id, bool host)
{
    Pool &p = host ? state().host[dev] : state().dev[dev];
    renew(p, id);
    return p;
}

cudaError_t alloc(void **p, size_t bytes, bool host)
{
    const auto fresh = [&](size_t size) {
        return host ? cudaHostAlloc(p, size, cudaHostAllocMapped) : cudaMalloc(p, size);
    };
    const size_t size = rounded(bytes);
    int dev;
    unsigned long long id;
    if (!where(&dev, &id))
        return fresh(bytes);
    State &s = state();
    size_t cap;
    {
        std::lock_guard<std::mutex> g(s.lock);
        Pool &pool = pool_of(dev, id, host);
        if ((*p = take(pool, size)))
            return cudaSuccess;
        cap = pool.cap;
    }
    if (!cap) {
        size_t free_bytes = 0, total = 0;
        if (host)
            total = 32 * kHostCap;
        else if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess)
            cudaGetLastError();
        cap = total / 32;
    }
    cudaError_t e = fresh(size);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        bool any;
        {
            Released out(host);
            std::lock_guard<std::mutex> g(s.lock);
            Pool &pool = pool_of(dev, id, host);
            any = !pool.kept.empty();
            drop(pool, pool.kept.size(), &out);
        }
        if (any)
            e = fresh(size);
    }
    if (e != cudaSuccess) {
        *p = nullptr;
        return e;
    }
    std::lock_guard<std::mutex> g(s.lock);
    Pool &pool = pool_of(dev, id, host);
    pool.cap = cap;
    pool.live[*p] = size;
    return cudaSuccess;
}

void give_back(void *p, bool host, bool keep)
{
    if (!p)
        return;
    Released out(host);
    int dev;
    unsigned long long id;
    if (!where(&dev, &id)) {
        out.blocks.push_back(Block{p, 0, 0});
        return;
    }
    std::lock_guard<std::mutex> g(state().lock);
    put(pool_of(dev, id, host), p, keep, &out);
}

}  // namespace

unsigned long long cuda_context_id()
{
    static const auto fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<CUresult (*)(CUcontext, unsigned long long *)>(f);
    }();
    unsigned long long id = 0;
    if (!fn)
        return 1;
    // (a thread that has made no runtime call yet has no current context)
    if (fn(nullptr, &id) != CUDA_SUCCESS && (cudaFree(nullptr) != cudaSuccess || fn(nullptr, &id) != CUDA_SUCCESS)) {
        cudaGetLastError();
        return 0;
    }
    return id;
}

cudaError_t pool_alloc(void **p, size_t bytes) { return alloc(p, bytes, false); }
void pool_free(void *p, bool keep) { give_back(p, false, keep); }
cudaError_t pool_host_alloc(void **p, size_t bytes) { return alloc(p, bytes, true); }
void pool_host_free(void *p, bool keep) { give_back(p, true, keep); }

void pool_loaded()
{
    Released dev_out(false), host_out(true);
    int dev;
    unsigned long long id;
    if (!where(&dev, &id))
        return;
    std::lock_guard<std::mutex> g(state().lock);
    age(pool_of(dev, id, false), &dev_out);
    age(pool_of(dev, id, true), &host_out);
}

size_t pool_trim()
{
    Released dev_out(false), host_out(true);
    int dev;
    unsigned long long id;
    if (!where(&dev, &id))
        return 0;
    std::lock_guard<std::mutex> g(state().lock);
    Pool &d = pool_of(dev, id, false), &h = pool_of(dev, id, true);
    const size_t bytes = d.kept_bytes + h.kept_bytes;
    drop(d, d.kept.size(), &dev_out);
    drop(h, h.kept.size(), &host_out);
    return bytes;
}

cudaError_t configure_once(int which, cudaError_t (*configure)())
{
    static std::mutex lock;
    static unsigned long long done[kMaxDevices][kConfigCount];
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return configure();
    const unsigned long long id = cuda_context_id();
    std::lock_guard<std::mutex> g(lock);
    if (id && done[dev][which] == id)
        return cudaSuccess;
    const cudaError_t r = configure();
    if (r == cudaSuccess)
        done[dev][which] = id;
    return r;
}

}  // namespace pwa
