// The batched half-sweep: one launch per colour covers many replicas (used by
// the batch API and the server).
#pragma once
#include <cstdint>

#include "ising_device.cuh"
#include "ising_internal.h"

namespace ising {

// Device descriptor of one replica for the current run.
struct BatchReplica {
    uint64_t* w0;
    uint64_t* w1;
    Geom g;
    PhiloxKeys rk;
    uint32_t thr0, thr1, all0, all1;
    uint64_t t_start;               // sweep counter before this run
    uint32_t nsweeps;               // sweeps in this run
    uint32_t every;                 // record interval
    uint32_t phase;                 // records after sweeps s with (phase + s) % every == 0
    unsigned long long* counts;     // record k -> counts[2k], counts[2k+1] (anti, up)
    uint32_t rounds;                // Philox rounds of the sweep draws (10 or the opt-in 7)
};

// A block's items: blockDim.x consecutive ones of one strip of a replica (see
// Strips in ising_device.cuh).
struct BatchTile {
    int rep;            // replica
    uint32_t first;     // first item of the tile in its strip
    uint32_t strip;     // the strip's first word | its words << 16
    uint32_t magic;     // item / words of the strip (strip_group)
};

// The tiles of replica `rep` of geometry g, `threads` items each.
template <typename Tiles>
inline void add_tiles(Tiles& tiles, int rep, const Geom& g, int threads)
{
    const Strips st = make_strips(g.W, kStripWords);
    const uint32_t groups = (uint32_t)((g.L + 3) / 4);
    for (uint32_t k = 0; k < st.n; ++k) {
        const bool last = k == st.n - 1;
        const uint32_t width = last ? st.last : st.width;
        for (uint32_t f = 0; f < groups * width; f += (uint32_t)threads)
            tiles.push_back({rep, f, k * st.width | width << 16, last ? st.magic_last : st.magic});
    }
}

// One half-sweep of colour C over every replica that still has sweeps to do
// in this run: block b works on tile b, as half_sweep_kernel on its items.  What
// it reads before the wait (the tile, the replica and the chunk's counter) no
// half-sweep writes.  ROUNDS: the Philox rounds of every replica (0: each
// replica's own, a runtime choice).  REC: 0 records after the sweeps the
// replica's phase and interval pick, 1 never records, 2 records after every
// sweep (colour 1, interval 1).  Fixing both when a launch allows it removes
// the other code paths from the kernel: measured on GB300, scan 1,246 -> 1,284
// and batched 1,262 -> 1,284 spin-updates/ns.
template <int C, int ROUNDS = 0, int REC = 0>
__global__ void __launch_bounds__(256, 3)
batch_half_sweep_kernel(const BatchReplica* __restrict__ reps, const BatchTile* __restrict__ tiles,
                        const uint32_t* __restrict__ chunk_base, uint32_t s_local)
{
    __shared__ uint2 tab[kFields * kStripWords];
    pdl_launch();
    const BatchTile tile = tiles[blockIdx.x];
    const BatchReplica* R = reps + tile.rep;
    const uint32_t s = *chunk_base + s_local;      // sweep of this run, 1-based
    if (s > R->nsweeps) {                          // uniform over the block
        pdl_wait();    // every block waits, so a grid that has completed implies all those before it
        return;
    }
    const Geom g = R->g;
    const uint32_t w0 = tile.strip & 0xffffu, width = tile.strip >> 16;
    const uint32_t q = tile.first + threadIdx.x;
    const uint32_t grp = strip_group(q, tile.magic);
    const uint32_t x = q - grp * width;
    const bool valid = grp * 4u < (uint32_t)g.L;
    const uint64_t t = R->t_start + s;
    const PhiloxKeys rk = R->rk;
    uint32_t anti = 0, up = 0;
    ItemMasks acc;
    first_products<kFields, kStripWords>(tab, w0, width, tile.magic, philox_first_key((uint32_t)t, rk));
    if (valid) {
        const FirstTable first = {tab + x};
        if (ROUNDS == 7 || (ROUNDS == 0 && R->rounds == 7))
            draw_item<7>(first, grp, t, C, rk, R->thr0, R->thr1, R->all0, R->all1, acc);
        else
            draw_item<10>(first, grp, t, C, rk, R->thr0, R->thr1, R->all0, R->all1, acc);
    }
    pdl_wait();
    uint64_t* own = C == 0 ? R->w0 : R->w1;
    const uint64_t* other = C == 0 ? R->w1 : R->w0;
    uint32_t record = 0;                            // record number + 1 of this sweep
    if (C == 1 && REC == 2) record = s;
    if (C == 1 && REC == 0) {
        const uint32_t ps = R->phase + s, n = ps / R->every;
        if (n * R->every == ps) record = n;
    }
    if (C == 1 && REC != 1 && record) {
        if (valid) apply_item<C, true, true>(own, other, g, grp, w0 + x, acc, anti, up);
        block_add_counts(R->counts + 2 * (size_t)(record - 1), anti, up);
    } else if (C == 0 || REC != 2) {
        if (valid) apply_item<C, true, false>(own, other, g, grp, w0 + x, acc, anti, up);
    }
}

static __global__ void batch_advance_kernel(uint32_t* chunk_base, uint32_t n)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) *chunk_base += n;
}

}  // namespace ising
