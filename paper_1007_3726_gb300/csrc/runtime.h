// Host runtime pieces shared by the translation units of libising (error
// text, allocator hook, thresholds, parameter validation).
#pragma once

#include "ising.h"

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

namespace ising {

// An NVTX range for the lifetime of the object (visible in Nsight timelines;
// without a tool attached a push / pop costs a few nanoseconds).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// Sets the calling thread's last-error text and returns st.
ising_status fail(ising_status st, const char *fmt, ...);
void clear_error();

// Device allocator in force when a handle is created (cudaMalloc by default,
// or the hook installed with ising_set_allocator).
struct Allocator {
    ising_alloc_fn alloc = nullptr;
    ising_free_fn free_fn = nullptr;
    void *ctx = nullptr;
    void *allocate(size_t bytes, cudaStream_t s) const;
    void release(void *p, cudaStream_t s) const;
    // Scratch and staging memory, used in the order of stream s: from the hook, or
    // from a pool per device that keeps at most kPoolKeeps bytes of what was
    // released, so that a handle that comes and goes does not map and unmap its scratch
    // (where there is no pool, or it has no room, from cudaMalloc).
    void *scratch(size_t bytes, cudaStream_t s) const;
    void release_scratch(void *p, cudaStream_t s) const;
};
constexpr size_t kPoolKeeps = 1ull << 30;
Allocator current_allocator();

// The scratch of one owner (a handle, a batch): allocated by a call that needs it, in use
// from scratch_begin to scratch_end, and kept for the owner's next call as long as nobody
// else needs the memory.  What idle owners keep is given back, the longest unused first,
// when all owners of a device together would hold more than a quarter of its memory
// (scratch_limit), and altogether when an allocation of the library fails.  Giving back
// is ordered behind the owner's work on its stream.
struct Scratch {
    Allocator alloc;
    cudaStream_t stream = nullptr;
    int device = 0;
    void *p = nullptr;
    size_t bytes = 0;
    uint64_t made = 0;      // which allocation it is: another number, other contents
    // under the book's lock
    bool busy = false;      // a call is queueing work that uses it
    bool pinned = false;    // a captured graph holds its address: never given back
    uint64_t used = 0;      // order of the last uses
};
// At least `need` bytes at s.p and in use; false when they are not to be had (refused, more
// than kPoolKeeps and half of the free memory, or the stream is being captured).
bool scratch_begin(Scratch &s, size_t need);
void scratch_end(Scratch &s);                // all work that uses it is queued
void scratch_pin(Scratch &s, bool pinned);
void scratch_drop(Scratch &s);               // the owner ends; its stream's work is done
size_t scratch_bytes(const Scratch &s);      // that it holds now
void scratch_give_back();                    // all idle scratch of the current device, and the pools
size_t scratch_limit(int device);

struct ScratchUse {
    Scratch *s = nullptr;
    bool begin(Scratch &x, size_t need)
    {
        if (s || !scratch_begin(x, need)) return false;
        s = &x;
        return true;
    }
    ScratchUse() = default;
    ~ScratchUse()
    {
        if (s) scratch_end(*s);
    }
    ScratchUse(const ScratchUse &) = delete;
    ScratchUse &operator=(const ScratchUse &) = delete;
};

// floor(2^32 exp(-dE / T)), clamped to [0, 2^32 - 1].
uint32_t threshold_for(double dE, double T);
bool valid_temperature(double T);

ising_status validate_params(const ising_params *p, uint32_t *word_bits);

}  // namespace ising
