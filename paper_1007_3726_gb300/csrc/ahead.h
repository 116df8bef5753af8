// The draw-ahead form of a sweep call (ahead.cu): its plan, the arguments of one
// launch and the launcher.
#pragma once

#include "kernels.h"

#include <cstddef>
#include <cstdint>

namespace ising {

struct AheadPlan {
    uint32_t kw;            // rows of a column that an update thread holds (2, 4 or 8); 0: no plan
    uint32_t tile_rows;     // rows of a tile
    uint32_t halo;          // redundant rows on either side of it (0: the tile is the lattice)
    uint32_t tiles;
    uint32_t update_ctas;   // CTAs that share them
    bool warp;              // one warp holds the lattice
    bool field;             // in a field: five mask planes
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
    uint32_t u_steps, u_step0;    // steps; index of the first in the call
    const uint64_t *src;
    uint64_t *dst;
    const char *u_masks;
    uint32_t *u_snaps;            // states after the counted sweeps (where the tile is the lattice)
    uint32_t u_phase;             // sweep index % record_every at the block's start
    uint32_t u_recs, u_slot0;     // samples of the block, slot of the first
    uint32_t u_slots, u_last;     // counted sweeps: u_recs, or one more; the call's last block
    // count: the snapshots of the block before
    uint32_t count_ctas, c_slots, c_recs, c_slot0, c_last;
    const uint32_t *c_snaps;
    // draw: d_sweeps sweeps from sweep index d_t0, in tickets of 32 items of 4 sweeps or of one
    uint32_t d_t0, d_sweeps, d_four, d_tickets;
    char *d_masks;
    unsigned int *d_ticket, *next_ticket;  // this launch's counter; the one to clear
};

AheadPlan ahead_plan(uint64_t L, bool field);

}  // namespace ising

struct ising_lattice;

namespace ising {
// The handle's scratch for the plan (masks, snapshots, a second lattice), allocated
// on first use and kept; false when there is none to be had (the allocator refuses,
// or the stream is being captured): the caller then takes another path.
bool ahead_ready(ising_lattice *h, const AheadPlan &pl);
// Queues nsweeps sweeps of `lattice` (the handle's, or a copy of it) from sweep
// index t0 on the handle's stream; counters as TinyRunArgs.  A block holds at most
// max_block sweeps.
cudaError_t ahead_sweeps(ising_lattice *h, const AheadPlan &pl, void *lattice, uint64_t t0, uint64_t nsweeps,
                         uint32_t record_every, uint64_t nrec, unsigned int *err, uint32_t hold_step, uint64_t max_block);
}  // namespace ising
