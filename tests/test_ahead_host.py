"""Host-side rules of the draw-ahead form (csrc/ahead.h) and of the memory it works in,
compiled with the host compiler and run without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1007_3726_gb300", "csrc")


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(d, "cuda_runtime.h")):
        pytest.skip("CUDA headers not found")
    return d


def _run(tmp_path, source, *files):
    """Compiles a C++ program against the library's headers (and some of its files) and
    returns what it prints."""
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(source)
    cmd = ["g++", "-std=c++17", "-g", "-fsanitize=undefined", "-fno-sanitize-recover=undefined", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
           _cuda_include(), "-o", str(exe), str(src)]
    for f in files:
        cmd += ["-x", "c++", os.path.join(CSRC, f)]
    r = subprocess.run([*cmd, "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return r.stdout


DRAW_GRID = r"""
#include "ahead.h"
#include <cstdio>
using namespace ising;
int main()
{
    const uint32_t T = 512;
    for (uint32_t sms = 1; sms <= 152; sms += sms < 70 ? 1 : 41)
        for (uint32_t L : {320u, 512u})
            for (uint32_t slots : {0u, 1u, 7u, 64u, 128u})
                for (uint32_t tickets : {0u, 1u, 200u, 8192u}) {
                    const uint32_t runs = L * (L / 64) / 2, per = (runs + 31u) & ~31u;
                    const DrawGrid g = draw_grid(sms, T, slots, runs, tickets);
                    // the kernel's loop: CTA c < count_ctas takes items c T + thread, in strides of count_ctas T
                    uint64_t done = 0;
                    for (uint32_t c = 0; c < g.grid && c < g.count_ctas; ++c)
                        for (uint64_t first = (uint64_t)c * T; first < (uint64_t)slots * per; first += (uint64_t)g.count_ctas * T)
                            done += std::min<uint64_t>(T, (uint64_t)slots * per - first);
                    if (done != (uint64_t)slots * per || g.grid < 1 || g.grid > sms) {
                        std::printf("sms %u L %u slots %u tickets %u: %llu of %llu counted by %u of %u CTAs\n", sms, L, slots, tickets,
                                    (unsigned long long)done, (unsigned long long)slots * per, g.grid, g.count_ctas);
                        return 1;
                    }
                }
    return 0;
}
"""


def test_every_snapshot_is_counted_on_any_number_of_sms(tmp_path):
    _run(tmp_path, DRAW_GRID)


# The CUDA runtime calls that memory.cu makes, over a device of 1000 MB in which a pool keeps
# what is freed until it is trimmed.
FAKE_CUDART = r"""
#include "runtime.h"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
using namespace ising;
constexpr size_t MB = 1 << 20, kTotal = 1000 * MB;
std::mutex mu;
std::map<void *, size_t> plain, pooled;
size_t pool_reserved = 0;
bool pools = true, fragmented = false;
cudaStream_t in_capture = nullptr;
std::vector<cudaStream_t> waited;
uintptr_t next_address = 4096;
size_t sum(const std::map<void *, size_t> &m) { size_t n = 0; for (auto &x : m) n += x.second; return n; }
size_t taken() { return sum(plain) + std::max(pool_reserved, sum(pooled)); }
void *fresh(size_t n) { void *p = (void *)next_address; next_address += n + 256; return p; }
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { std::lock_guard<std::mutex> l(mu); *f = kTotal - taken(); *t = kTotal; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n)
{
    std::lock_guard<std::mutex> l(mu);
    if (taken() + n > kTotal) return cudaErrorMemoryAllocation;
    plain[*p = fresh(n)] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { std::lock_guard<std::mutex> l(mu); if (!plain.erase(p) && !pooled.erase(p)) std::abort(); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { if (!pools) return cudaErrorNotSupported; *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void *v)
{
    std::lock_guard<std::mutex> l(mu);
    *(uint64_t *)v = a == cudaMemPoolAttrReservedMemCurrent ? pool_reserved : sum(pooled);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { std::lock_guard<std::mutex> l(mu); pool_reserved = sum(pooled); return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t)
{
    std::lock_guard<std::mutex> l(mu);
    const size_t reserved = fragmented ? pool_reserved + n : std::max(pool_reserved, sum(pooled) + n);
    if (sum(plain) + reserved > kTotal) return cudaErrorMemoryAllocation;
    pool_reserved = reserved;
    pooled[*p = fresh(n)] = n;
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { std::lock_guard<std::mutex> l(mu); if (!pooled.erase(p)) std::abort(); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { std::lock_guard<std::mutex> l(mu); waited.push_back(s); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *c)
{
    *c = in_capture && s == in_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
cudaStream_t stream(int k) { return (cudaStream_t)(uintptr_t)(k + 1); }
"""

SCRATCH_BOOK = FAKE_CUDART + r"""
// a hook over 500 MB of its own that comes back into the library when it frees
size_t hook_held = 0;
std::map<void *, size_t> hooked;
Scratch *reenter = nullptr;
void *hook_alloc(size_t n, void *, void *) { if (hook_held + n > 500 * MB) return nullptr; void *p = fresh(n); hooked[p] = n; hook_held += n; return p; }
void hook_free(void *p, void *, void *)
{
    if (!hooked.count(p)) std::abort();
    hook_held -= hooked[p];
    hooked.erase(p);
    if (reenter) { Scratch *s = reenter; reenter = nullptr; scratch_drop(*s); }
}
bool call(Scratch &s, size_t n) { if (!scratch_begin(s, n)) return false; scratch_end(s); return true; }
int main()
{
    // in all at most a quarter of the device, the longest unused gives way
    Scratch s[20];
    for (int k = 0; k < 20; ++k) s[k].stream = stream(k);
    for (int k = 0; k < 20; ++k) {
        CHECK(call(s[k], 60 * MB));
        CHECK(sum(pooled) <= kTotal / 4);
    }
    for (int k = 0; k < 20; ++k) CHECK((s[k].p != nullptr) == (k >= 16));
    CHECK(call(s[16], 50 * MB) && sum(pooled) == 240 * MB);      // there already
    CHECK(call(s[0], 60 * MB) && s[16].p && !s[17].p);           // 17 is the longest unused now
    // one in use, or in a captured graph, stays; its owner gets no larger one while captured
    CHECK(scratch_begin(s[18], 60 * MB));
    in_capture = stream(19);
    CHECK(call(s[19], 60 * MB) && !scratch_begin(s[19], 70 * MB) && s[19].bytes == 60 * MB);
    in_capture = nullptr;
    CHECK(!scratch_begin(s[19], 70 * MB));
    CHECK(call(s[1], 240 * MB) && s[18].p && s[19].p && !s[0].p && !s[16].p);
    scratch_give_back();
    CHECK(!s[1].p && s[18].p && s[19].p && sum(pooled) == 120 * MB && pool_reserved == 120 * MB);
    scratch_end(s[18]);
    // an allocation that would fail takes what is idle, and nothing else
    CHECK(call(s[2], 100 * MB));
    Allocator al;
    void *big = al.allocate(930 * MB, nullptr);
    CHECK(big && !s[2].p && !s[18].p && s[19].p);
    CHECK(!al.allocate(100 * MB, nullptr) && !al.scratch(100 * MB, nullptr));
    CHECK(!call(s[3], 20 * MB) && !s[3].p);
    al.release(big, nullptr);
    CHECK(call(s[3], 20 * MB));
    // staging memory that the pool has no piece for comes from elsewhere, once what the
    // pool keeps has been trimmed, and goes back there
    pool_reserved = 900 * MB;
    fragmented = true;
    void *st = al.scratch(400 * MB, nullptr);
    CHECK(st && sum(plain) == 400 * MB && pool_reserved == 60 * MB && !s[3].p);
    al.release_scratch(st, nullptr);
    CHECK(plain.empty());
    fragmented = false;
    // hooks: released without the lock, after their stream has been waited for
    Scratch h[3];
    for (int k = 0; k < 3; ++k) { h[k].alloc = Allocator{hook_alloc, hook_free, nullptr}; h[k].stream = stream(100 + k); }
    CHECK(call(h[0], 80 * MB) && call(h[1], 80 * MB) && h[0].p);
    waited.clear();
    reenter = &h[1];
    CHECK(call(h[2], 200 * MB) && !h[0].p && !h[1].p && hook_held == 200 * MB);
    CHECK(!waited.empty() && waited[0] == stream(100));
    void *l = h[0].alloc.allocate(450 * MB, nullptr);
    CHECK(l && !h[2].p && hook_held == 450 * MB);
    h[0].alloc.release(l, nullptr);
    // owners that come, work and go on several threads, close to the limit
    scratch_drop(s[19]);
    std::vector<std::thread> th;
    bool ok[8];
    for (int t = 0; t < 8; ++t)
        th.emplace_back([t, &ok] {
            ok[t] = true;
            for (int i = 0; i < 400; ++i) {
                Scratch a, b;
                a.stream = stream(200 + t);
                b.stream = stream(300 + t);
                for (int k = 0; k < 3; ++k) {
                    if (scratch_begin(a, (20 + k) * MB)) { ok[t] = ok[t] && a.p && a.bytes >= (20 + k) * MB; scratch_end(a); } else ok[t] = false;
                    if (!call(b, 40 * MB)) ok[t] = false;
                }
                if (i % 50 == 0) scratch_give_back();
                scratch_drop(a);
                scratch_drop(b);
            }
        });
    for (auto &x : th) x.join();
    for (bool o : ok) CHECK(o);
    for (Scratch &x : s) scratch_drop(x);
    for (Scratch &x : h) scratch_drop(x);
    CHECK(pooled.empty() && plain.empty() && hooked.empty());
    return 0;
}
"""


def test_scratch_is_bounded_and_given_back(tmp_path):
    _run(tmp_path, SCRATCH_BOOK, "memory.cu")


NO_POOL = FAKE_CUDART + r"""
int main()
{
    // a device without memory pools: staging memory still comes, scratch does not
    pools = false;
    Allocator al;
    void *st = al.scratch(100 * MB, nullptr);
    CHECK(st && sum(plain) == 100 * MB);
    al.release_scratch(st, nullptr);
    CHECK(plain.empty());
    Scratch s;
    CHECK(!scratch_begin(s, MB) && !s.p && plain.empty());
    return 0;
}
"""


def test_staging_memory_without_memory_pools(tmp_path):
    _run(tmp_path, NO_POOL, "memory.cu")
