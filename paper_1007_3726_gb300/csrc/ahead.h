// The draw-ahead form of a sweep call (ahead.cu): its plan, the arguments of one
// launch and the launcher.
#pragma once

#include "kernels.h"

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace ising {

struct AheadPlan {
    uint32_t kw;            // rows of a column that an update thread holds (2, 4 or 8); 0: no plan
    uint32_t tile_rows;     // rows of a tile
    uint32_t halo;          // redundant rows on either side of it (0: the tile is the lattice)
    uint32_t tiles;
    uint32_t update_ctas;   // CTAs that share them
    bool warp;              // one warp holds the lattice
    bool cluster;           // the CTAs of one cluster hold it
    uint32_t stages;        // and have the masks of that many chunks of steps in shared memory
    bool field;             // in a field: five mask planes
    bool two;               // two CTAs share a SM
    uint32_t band_rows;     // rows that a launch takes (0: all)
    uint32_t tile_words, tiles_x;  // words of a tile's rows and tiles of a row, where a launch takes a band
    uint32_t block_sweeps;  // sweeps of a block at most (halo / 2 where there is a halo)
    uint32_t min_sweeps;    // shorter calls are as fast without
    uint32_t step_bytes;    // masks of a step
    size_t mask_bytes;      // one buffer of masks
    size_t snap_bytes;      // one buffer of snapshots
};

// x / d for x < 2^24 by a multiplication: mul = ceil(2^shift / d), 2^(shift - 24) >= d.
struct FastDiv {
    uint32_t mul, shift;
    __host__ __device__ uint32_t quotient(uint32_t x) const { return (uint32_t)(((uint64_t)x * mul) >> shift); }
};

// The arguments of one launch.
struct AheadArgs {
    RoundKeys key;
    uint32_t thr[5], c3base;      // thresholds of the mask planes: P4 and P8, or the five in a field
    uint32_t plus3, plus4, minus0, minus1, flipped;  // in a field (step_run_field)
    uint32_t L, wc, nwords;       // words per row and in all, of one colour
    FastDiv by_wc, by_group;      // divisions by wc and nwords / 32
    uint32_t step_bytes;          // of a step's masks
    uint32_t record_every;        // 0: record nothing
    unsigned long long *acc, *final_acc;
    unsigned int *err;            // set when a wait ran out
    uint32_t hold_step;           // failure testing: 1 + a step whose masks never arrive
    // update: u_steps steps (0: none) from src to dst
    uint32_t update_ctas, tiles, tile_rows, halo;
    uint32_t stages;              // chunks of masks in shared memory (cluster form)
    uint32_t u_steps, u_step0;    // steps; index of the first in the call
    const uint64_t *src;
    uint64_t *dst;
    const char *u_masks;
    uint32_t *u_snaps;            // states after the counted sweeps
    uint32_t u_phase;             // sweep index % record_every at the block's start
    uint32_t u_recs, u_slot0;     // samples of the block, slot of the first
    uint32_t u_slots, u_last;     // counted sweeps: u_recs, or one more; the call's last block
    // a band of rows: its first; the first row and the words of a step with masks
    uint32_t u_row0, u_mask_row0, u_words;
    uint32_t tile_words, tiles_x;
    FastDiv by_tw;                // division by tile_words + 2
    // count: the snapshots of the block before
    uint32_t count_ctas, c_slots, c_recs, c_slot0, c_last;
    uint32_t c_wait;              // they are those of the launch before
    // cluster form: updates of the call whose writes are visible (each publishes those before
    // it); those before this update; those that a draw launch needs (0: it waits, or none)
    unsigned int *done;
    uint32_t u_before, d_after;
    const uint32_t *c_snaps;
    // draw: d_sweeps sweeps from sweep index d_t0, in tickets of 32 items of d_k sweeps
    uint32_t d_t0, d_sweeps, d_k, d_tickets;
    uint32_t d_row0, d_words;     // a band: the first row drawn, words of a step
    char *d_masks;
    unsigned int *d_ticket, *next_ticket;  // this launch's counter; the one to clear
};

// A launch of the cluster form's draws and counts.
struct DrawGrid {
    uint32_t count_ctas, grid;  // CTAs that count (the first ones), and in all
};
// For `slots` snapshots of `runs` runs and `tickets` items, with CTAs of `threads` threads
// on `sms` SMs (one CTA each).  The counting CTAs share the snapshots by their number, so
// that all of them have to be in the grid, also on a partition with few SMs.
inline DrawGrid draw_grid(uint32_t sms, uint32_t threads, uint32_t slots, uint32_t runs, uint32_t tickets)
{
    const uint32_t per = (runs + 31u) & ~31u;  // threads a snapshot: whole warps
    DrawGrid g;
    g.count_ctas = std::min({(slots * per + threads - 1) / threads, 64u, sms});
    g.grid = std::max(1u, std::min(sms, g.count_ctas + (tickets + threads / 32u - 1) / (threads / 32u)));
    return g;
}

AheadPlan ahead_plan(uint64_t L, bool field);
// The cluster form, for the sizes and calls where it is the faster one (no field; kw 0: not
// here).
AheadPlan cluster_plan(uint64_t L, uint64_t nsweeps);

// One lattice of a batch run (device table).
struct AheadJob {
    RoundKeys key;
    uint32_t thr[5], c3base;
    uint32_t plus3, plus4, minus0, minus1, flipped;
    uint32_t L, wc, nwords;
    FastDiv by_wc, by_group;
    uint32_t step_bytes, record_every;
    uint32_t field, kw, tile_rows, halo;
    uint32_t sweeps, block_sweeps, nblocks;   // of the run; of a block; blocks of the run
    uint32_t index;                           // of the lattice in the batch
    uint32_t tile_start, ticket_start;        // tiles and tickets of the jobs before
    size_t mask_bytes;                        // one buffer of masks
    char *masks;
    uint64_t *even, *odd;                     // the lattice before blocks 0, 2, .. and before blocks 1, 3, ..
    const uint64_t *copy_from;                // where `even` is not the lattice: copied from here first
    unsigned long long *acc, *final_acc;
};

struct AheadBatchArgs {
    const AheadJob *jobs;
    const uint32_t *t0;           // first sweep index of each lattice
    uint32_t block;               // drawn by this launch; the one before is updated
    uint32_t d_jobs, u_jobs;      // jobs that have them
    uint32_t d_tickets, u_tiles, update_ctas;
    unsigned int *d_ticket, *next_ticket;
    unsigned int *done;           // 1 once the run's first launch has waited for what was before it
    unsigned int *err;
};

}  // namespace ising

struct ising_lattice;

namespace ising {
// Bytes of scratch that the plan of size L works in (masks, snapshots, a second lattice).
size_t ahead_bytes(const AheadPlan &pl, uint64_t L);
// Queues nsweeps sweeps of `lattice` (the handle's, or scratch of L^2 sites) from sweep
// index t0 on the handle's stream, in its scratch; counters as TinyRunArgs.  A block holds at most
// max_block sweeps.
cudaError_t ahead_sweeps(ising_lattice *h, const AheadPlan &pl, void *lattice, uint64_t L, uint64_t t0,
                         uint64_t nsweeps, uint32_t record_every, uint64_t nrec, unsigned int *err, uint32_t hold_step, uint64_t max_block);

// A run of many lattices in the draw-ahead form.
struct AheadBatch {
    std::vector<AheadJob> jobs;   // by falling number of blocks
    uint32_t total_tiles = 0, total_tickets = 0;
    size_t smem = 0, table_bytes = 0, scratch_bytes = 0;
    char *d_scratch = nullptr;
    // Plans runs of sweeps[i] sweeps of hs[i]; false if a lattice has no tiles.
    bool plan(const std::vector<ising_lattice *> &hs, const std::vector<uint64_t> &sweeps,
              const std::vector<uint32_t> &record_every);
    // Places the jobs in scratch (scratch_bytes) and uploads their table.
    cudaError_t upload(void *scratch, const std::vector<ising_lattice *> &hs, const std::vector<unsigned long long *> &acc,
                       const std::vector<unsigned long long *> &final_acc, cudaStream_t s);
    // Queues one run; d_t0: the lattices' first sweep indices on the device, d_err: its error
    // flag.
    cudaError_t enqueue(const uint32_t *d_t0, unsigned int *d_err, cudaStream_t s);
};
}  // namespace ising
