// Device memory of the library: the allocator hook or cudaMalloc, the pool that scratch and
// staging memory comes from, and the book of the scratch that owners keep between calls.
// Host code only.
#include "runtime.h"

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <mutex>
#include <set>
#include <vector>

namespace ising {

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};
std::set<void *> g_plain;  // staging memory from cudaMalloc

// The scratch pool of the current device, made on first use; nullptr if there is none.
cudaMemPool_t device_pool()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        uint64_t keeps = kPoolKeeps;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess ||
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keeps) != cudaSuccess) {
            cudaGetLastError();
            if (pool) cudaMemPoolDestroy(pool);
            return nullptr;
        }
        g_pool[dev] = pool;
    }
    return g_pool[dev];
}

// Gives back what the pools of all devices keep unused.
void trim_pools()
{
    std::lock_guard<std::mutex> lk(g_pool_mu);
    for (cudaMemPool_t p : g_pool)
        if (p) cudaMemPoolTrimTo(p, 0);
}

// Bytes that an allocation from the pool may take: the device's free memory and what the
// pool keeps unused.  0 if it cannot be told.
size_t available_bytes()
{
    size_t free_bytes = 0, total_bytes = 0;
    if (cudaMemGetInfo(&free_bytes, &total_bytes) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    uint64_t reserved = 0, used = 0;
    const cudaMemPool_t pool = device_pool();
    if (pool && cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) == cudaSuccess &&
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess && reserved > used)
        free_bytes += reserved - used;
    return free_bytes;
}

void *from_pool(size_t bytes, cudaStream_t s)
{
    const cudaMemPool_t pool = device_pool();
    void *p = nullptr;
    if (pool && cudaMallocFromPoolAsync(&p, bytes ? bytes : 16, pool, s) == cudaSuccess) return p;
    cudaGetLastError();
    return nullptr;
}

// ---------------------------------------------------------------- the book --
std::mutex g_book_mu;
std::set<Scratch *> g_held;  // owners with memory
uint64_t g_use = 0;          // uses and allocations, counted

struct HookFree {
    Allocator alloc;
    void *p;
    cudaStream_t s;
};

bool capturing(cudaStream_t s)
{
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) == cudaSuccess) return cap != cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return true;
}

// What idle owners of the device keep.
size_t idle_bytes(int device)
{
    size_t n = 0;
    for (const Scratch *s : g_held)
        if (s->device == device && !s->busy && !s->pinned) n += s->bytes;
    return n;
}

// Takes the memory of idle owners of the device, the longest unused first, until the owners
// hold `most` bytes or less.  With `wait`, the memory is free when this returns.  Memory of
// hooks is idle then too and is left to the caller, to be released without the lock: a hook
// may come back into the library.
bool take_idle(int device, size_t most, bool wait, std::vector<HookFree> &hooks)
{
    std::vector<Scratch *> idle;
    size_t held = 0;
    for (Scratch *s : g_held)
        if (s->device == device) {
            held += s->bytes;
            if (!s->busy && !s->pinned) idle.push_back(s);
        }
    std::sort(idle.begin(), idle.end(), [](const Scratch *x, const Scratch *y) { return x->used < y->used; });
    bool any = false;
    for (Scratch *s : idle) {
        if (held <= most) break;
        if (capturing(s->stream)) continue;
        if (s->alloc.free_fn) {
            cudaStreamSynchronize(s->stream);
            hooks.push_back(HookFree{s->alloc, s->p, s->stream});
        } else {
            s->alloc.release_scratch(s->p, s->stream);
            if (wait) cudaStreamSynchronize(s->stream);
        }
        held -= s->bytes;
        s->p = nullptr;
        s->bytes = 0;
        g_held.erase(s);
        any = true;
    }
    return any;
}

// All idle scratch of the current device; whether there was any.
bool take_all_idle()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::vector<HookFree> hooks;
    bool any;
    {
        std::lock_guard<std::mutex> lk(g_book_mu);
        any = take_idle(dev, 0, true, hooks);
    }
    for (const HookFree &f : hooks) f.alloc.release_scratch(f.p, f.s);
    return any;
}
}  // namespace

void *Allocator::allocate(size_t bytes, cudaStream_t s) const
{
    if (bytes == 0) bytes = 16;
    for (int attempt = 0; attempt < 2; ++attempt) {
        void *p = nullptr;
        if (alloc) {
            if ((p = alloc(bytes, (void *)s, ctx)) != nullptr) return p;
        } else {
            if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
            cudaGetLastError();  // clear the (non-sticky) allocation error
        }
        if (attempt == 0) {
            const bool any = take_all_idle();
            if (alloc && !any) break;
            trim_pools();
        }
    }
    return nullptr;
}

void Allocator::release(void *p, cudaStream_t s) const
{
    if (!p) return;
    if (free_fn)
        free_fn(p, (void *)s, ctx);
    else
        cudaFree(p);
}

void *Allocator::scratch(size_t bytes, cudaStream_t s) const
{
    if (alloc) return allocate(bytes, s);
    if (void *p = from_pool(bytes, s)) return p;
    void *p = allocate(bytes, s);  // no pool, or it is full: what is idle goes, the pools are trimmed
    if (p) {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        g_plain.insert(p);
    }
    return p;
}

void Allocator::release_scratch(void *p, cudaStream_t s) const
{
    if (!p) return;
    if (free_fn) {
        free_fn(p, (void *)s, ctx);
        return;
    }
    bool plain;
    {
        std::lock_guard<std::mutex> lk(g_pool_mu);
        plain = g_plain.erase(p) != 0;
    }
    if (!plain && cudaFreeAsync(p, s) == cudaSuccess) return;
    cudaGetLastError();
    cudaFree(p);
}

size_t scratch_limit(int device)
{
    if (const char *e = std::getenv("ISING_SCRATCH_MB"))  // testing only
        return (size_t)std::strtoull(e, nullptr, 10) << 20;
    // (asked for once a device)
    static std::atomic<size_t> total[kMaxDevices];
    const bool cached = device >= 0 && device < kMaxDevices;
    size_t n = cached ? total[device].load(std::memory_order_relaxed) : 0, free_bytes = 0;
    if (n == 0) {
        if (cudaMemGetInfo(&free_bytes, &n) != cudaSuccess) cudaGetLastError();
        if (cached) total[device].store(n, std::memory_order_relaxed);
    }
    return n / 4;
}

bool scratch_begin(Scratch &s, size_t need)
{
    const bool cap = capturing(s.stream);
    std::vector<HookFree> hooks;
    bool fits = true;
    {
        std::lock_guard<std::mutex> lk(g_book_mu);
        s.used = ++g_use;
        if (s.p && s.bytes >= need) {
            s.busy = true;
            s.pinned = s.pinned || cap;
            return true;
        }
        // nothing is allocated while the stream is captured, and what a graph holds stays
        if (cap || s.pinned) return false;
        if (s.p) {
            g_held.erase(&s);
            if (s.alloc.free_fn) {
                cudaStreamSynchronize(s.stream);
                hooks.push_back(HookFree{s.alloc, s.p, s.stream});
            } else {
                s.alloc.release_scratch(s.p, s.stream);
            }
            s.p = nullptr;
            s.bytes = 0;
        }
        const size_t most = scratch_limit(s.device);
        take_idle(s.device, most > need ? most - need : 0, false, hooks);
        // a second copy of a lattice that fills the GPU would take what its user may need:
        // at most half of what is free, and rather that than what idle owners keep
        if (need > kPoolKeeps) {
            const size_t available = available_bytes();
            fits = need <= available / 2;
            if (!fits && need <= (available + idle_bytes(s.device)) / 2) take_idle(s.device, 0, true, hooks);
        }
    }
    for (const HookFree &f : hooks) f.alloc.release_scratch(f.p, f.s);
    if (!fits && need > available_bytes() / 2) return false;
    void *p = s.alloc.alloc ? s.alloc.allocate(need, s.stream) : from_pool(need, s.stream);
    if (!p && !s.alloc.alloc && take_all_idle()) {
        trim_pools();
        p = from_pool(need, s.stream);
    }
    if (!p) return false;
    std::lock_guard<std::mutex> lk(g_book_mu);
    s.p = p;
    s.bytes = need;
    s.made = ++g_use;
    s.busy = true;
    g_held.insert(&s);
    return true;
}

void scratch_end(Scratch &s)
{
    std::lock_guard<std::mutex> lk(g_book_mu);
    s.busy = false;
}

void scratch_pin(Scratch &s, bool pinned)
{
    std::lock_guard<std::mutex> lk(g_book_mu);
    s.pinned = pinned;
}

void scratch_drop(Scratch &s)
{
    void *p;
    {
        std::lock_guard<std::mutex> lk(g_book_mu);
        p = s.p;
        g_held.erase(&s);
        s.p = nullptr;
        s.bytes = 0;
        s.busy = s.pinned = false;
    }
    s.alloc.release_scratch(p, s.stream);
}

size_t scratch_bytes(const Scratch &s)
{
    std::lock_guard<std::mutex> lk(g_book_mu);
    return s.bytes;
}

void scratch_give_back()
{
    take_all_idle();
    trim_pools();
}

}  // namespace ising
