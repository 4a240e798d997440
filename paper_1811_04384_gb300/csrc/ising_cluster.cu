// Cluster-resident temporal blocking for mid-size lattices (above the on-chip
// range, L of about 130 to 3000): rows of more than 14 dense words, and several
// clusters; one cluster on shorter rows is ising_band.cu's.
//
// There a half-sweep is short: a launch per half-sweep costs more than its
// work.  Here one launch of G thread-block clusters (of 16 blocks where the
// device allows it, else 8) runs a piece of up to 256 sweeps whose accept
// masks dense_mask_draw_kernel draws on the SMs the clusters leave free.  The
// launch's G C blocks own consecutive row bands of both colours, block B rows
// B L / (G C) .. (B + 1) L / (G C) - 1, and keep them in shared memory for the
// whole launch in the dense form of ising_dense.cuh (one bit per spin), in a
// window with k rows of halo above and below (k even, k <= kClHalo, k <= the
// rows a block owns, so a halo lies in the two neighbouring blocks).  The
// launch's half-sweeps run in phases of k:
//   1. each block takes the halo rows its neighbours pushed at the end of the
//      phase before (two sets of slots, by phase parity);
//   2. k half-sweeps on the window: after half-sweep d (0-based) the window
//      rows 1 + d .. R - 2 - d are exact, so after k of them the block's own
//      rows still are (a trapezoid: the halo rows are recomputed by both
//      neighbours);
//   3. each block pushes its first and last k own rows to the blocks above
//      and below: into their shared memory inside a cluster (distributed
//      shared memory), through a small global buffer with release/acquire
//      sequence flags between clusters;
//   4. a cluster barrier.
// Every thread updates the same 1 or 2 units (V = 1 or 2 dense words) in each
// half-sweep (those inside its trapezoid), with their offsets worked out once
// per launch, and copies their masks asynchronously into its own slots of
// shared memory, DEPTH half-sweeps ahead (no other thread reads them, so they
// need no barrier; as loads into registers that far ahead they waited for one
// another: 889 against 614 us for 1000 sweeps of L = 296).  The lattice's own words are converted as a launch starts and ends; a
// launch can also take its rows from a dense array (the column-interleaved
// layout's scratch).
//
// What bounds it: with 3-bit fields in the window the update itself did (101
// warp instructions per warp and half-sweep for 32 x 21 sites, on 16 to 96
// SMs), and more clusters left fewer SMs for the draws.  Dense words take
// about a tenth of the instructions per site, so from L of about 1100 the draws
// on the other SMs bound the path, and below that the latency of a half-sweep
// (mask wait, block barrier, shared-memory round trip) does as well: about 1,050 cycles
// at L = 1008.
//
// A wait between clusters that gives up (see cl_wait_flag in
// ising_cluster.cuh) lets the launch end with void results, and the host
// reports the failure.  Records (colour 1 of a recorded sweep) count each
// block's own rows only: every bond and spin once.
#include <cuda_runtime.h>
#include <cooperative_groups.h>

#include <algorithm>

#include "ising_cluster.cuh"
#include "ising_dense.cuh"
#include "ising_device.cuh"
#include "ising_internal.h"
#include "ising_per_device.h"

namespace cg = cooperative_groups;

namespace ising {
namespace {

constexpr int kClThreads = 1024;           // most threads of a block
// Most half-sweeps per phase.  A phase's exchange costs about 0.85 us, its halo
// rows are extra work: measured on GB300 (us of 1000 sweeps, record every 10, k
// = 8 / 12 / 18 / 24) L = 296: 610 / 565 / 544 / 543; L = 512: 713 / 688 / 652 /
// 641; L = 1008 (500 sweeps): 666 / 640 / 615 / 615; but L = 1700 (400 sweeps, two
// clusters) 12 / 18: 991 / 1023; L = 2600 (200, four): 1,028 / 1,042.
constexpr int kClHalo = 18, kClHaloWide = 12, kClWideWords = 21;   // 12 from rows of more than 21 words (L > 1344)
// Up to this many window words: one word per unit (one cluster, before short
// rows had their own form: L = 512 688 us against 846 with two, L = 700, above it:
// 872 with two against 982).  Since then: small windows of several clusters, and
// L <= 128 on this path.
constexpr long long kClOneWord = 512;

struct ClusterArgs {
    uint64_t* w[2];             // the lattice's colour arrays, L x g.P words each (null: `dense`)
    uint32_t* dense;            // or a dense array, [colour][row][word], L x d.P words per colour
    Geom g;
    DenseGeom d;
    int k;                      // half-sweeps per phase = halo rows
    int nsweeps;                // sweeps of this launch
    int rmax;                   // window rows the shared memory holds (largest share of rows + 2 k)
    const uint64_t* masks;      // masks[(h * L + i) * d.P + w]: half-sweep h = 2 j + c of the launch, row i, word w
    int64_t s0;                 // the launch runs sweeps s0 + 1 .. s0 + nsweeps of the call
    int64_t every;              // record after sweeps s with s % every == 0 (0: none)
    unsigned long long* counts; // count slots; record r of the call -> slots r `slots` ..
    int slots;                  // of a record, a power of two
    int G;                      // clusters of the launch: blocks g C .. g C + C - 1 form cluster g
    uint64_t* xbuf;             // G > 1: halo rows between clusters, [boundary][dir][parity][colour], k x d.P / 2 words
    unsigned long long* xflag;  // G > 1: [boundary][dir] sequence flags
    unsigned long long xseq;    // push m of this launch sets its flags to xseq + m + 1
    unsigned long long xwait;   // added to the values the receives wait for (0; a test stalls with more)
    unsigned int* xerr;         // set to 1 when a wait for a flag gives up
    unsigned int* gate;         // G > 1: the words the blocks agree through (cl_count_in, cl_decide)
    unsigned int gate_blocks;   // blocks that must have counted in (the launch's; one more in a test)
    unsigned int piece;         // the launch's number among those that agree
};

// Shared memory by 32-bit address: a half-sweep is short, and with generic
// 64-bit pointers its address arithmetic took as many instructions as the
// update.  `lo`, `hi` bound the array the access belongs to (checked build).
template <int V>
__device__ __forceinline__ void sh_ld(uint32_t addr, uint32_t (&x)[V], uint32_t lo, uint32_t hi, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index((addr - lo) / 4u + (V - 1), (hi - lo) / 4u, line)) {
        for (int j = 0; j < V; ++j) x[j] = 0;
        return;
    }
#endif
    if constexpr (V == 1) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x[0]) : "r"(addr));
    if constexpr (V == 2) asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x[0]), "=r"(x[1]) : "r"(addr));
    if constexpr (V == 4)
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(addr));
}

template <int V>
__device__ __forceinline__ void sh_st(uint32_t addr, const uint32_t (&x)[V], uint32_t lo, uint32_t hi, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index((addr - lo) / 4u + (V - 1), (hi - lo) / 4u, line)) return;
#endif
    if constexpr (V == 1) asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(x[0]) : "memory");
    if constexpr (V == 2) asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(x[0]), "r"(x[1]) : "memory");
}

// A unit (V dense words of a window row) a thread updates in every half-sweep
// whose rows include its row, with what the two colours need worked out once
// per launch.  The neighbour to the side of a site of colour C in global row i
// is at m - 1 when (i + C) is even, else m + 1: the other colour's row shifted
// by one bit, whose missing bit comes from the side word (the word before the
// unit, wrapped around the row, or the one after).  Across the wrap the bit is
// not at the word's end: to the left the last word is first shifted up by 32 -
// lb, to the right word 0's bit is placed at bit lb - 1 by a multiply.
struct Slot {
    int depth;            // half-sweeps of a phase the unit's row takes part in, less one; -1: no unit
    uint32_t at[2];       // shared address of the unit in the window of colour 0 and 1
    uint32_t side[2];     // and of the other colour's side word, for an update of colour 0 and 1
    uint32_t shl, mul;    // of the left and right side word across the wrap
    bool left0, own;      // colour 0 takes the left neighbour; an own row of the block
    bool last;            // the unit holds the row's last word
};

// One update of colour C with the masks m (flip_all; on dead
// bits and pad words the own spins, the vertical and the same-column neighbours
// and both masks are zero, so they never flip).  win0, win_bytes: shared
// address and bytes of a window (checked build); P4 the bytes of a row.  RECORD
// adds the unit's anti-aligned bonds and up spins over the live bits.  last_lo: the
// row's last word is the low word of its unit.
template <int V, int C, bool RECORD>
__device__ __forceinline__ void cl_update(const uint32_t (&m)[2 * V], uint32_t win0, uint32_t win_bytes, uint32_t P4,
                                          const Slot& sl, bool last_lo, uint32_t live_last, uint32_t& anti,
                                          uint32_t& up)
{
    const bool left = sl.left0 != (C == 1);
    const uint32_t a = sl.at[1 - C], own = win0 + C * win_bytes, other = win0 + (1 - C) * win_bytes;
    uint32_t s[V], u[V], d[V], h0[V], h1[V], sn[V], side[1];
    sh_ld<V>(a, h0, other, other + win_bytes, __LINE__);
    sh_ld<1>(sl.side[C], side, other, other + win_bytes, __LINE__);
    sh_ld<V>(a - P4, u, other, other + win_bytes, __LINE__);
    sh_ld<V>(a + P4, d, other, other + win_bytes, __LINE__);
    sh_ld<V>(sl.at[C], s, own, own + win_bytes, __LINE__);
    const uint32_t before = side[0] << sl.shl;
    if constexpr (V == 1) {
        const uint32_t r = __funnelshift_r(h0[0], side[0], 1) + side[0] * sl.mul;
        h1[0] = left ? __funnelshift_l(before, h0[0], 1) : r;
    } else {
        const uint32_t r0 = __funnelshift_r(h0[0], h0[1], 1) + side[0] * (last_lo ? sl.mul : 0u);
        const uint32_t r1 = __funnelshift_r(h0[1], side[0], 1) + side[0] * (last_lo ? 0u : sl.mul);
        h1[0] = left ? __funnelshift_l(before, h0[0], 1) : r0;
        h1[1] = left ? __funnelshift_l(h0[0], h0[1], 1) : r1;
    }
#pragma unroll
    for (int j = 0; j < V; ++j) sn[j] = flip_all(s[j], u[j], d[j], h0[j], h1[j], m[2 * j], m[2 * j + 1]);
    sh_st<V>(sl.at[C], sn, own, own + win_bytes, __LINE__);
    if (RECORD) {
#pragma unroll
        for (int j = 0; j < V; ++j) {
            // on the pad word of the last unit sn and h0 are zero and live must be
            const uint32_t live = !sl.last ? 0xffffffffu
                                           : (V == 1 || (j == 0) == last_lo ? live_last : (last_lo ? 0u : 0xffffffffu));
            anti += __popc(sn[j] ^ u[j]) + __popc(sn[j] ^ d[j]) + __popc(sn[j] ^ h0[j])
                  + __popc((sn[j] ^ h1[j]) & live);
            up += __popc(sn[j]) + __popc(h0[j]);
        }
    }
}

// Draws of at most this many threads (one a dense word and sweep), which leave
// most SMs idle for a chain of 64 calls, go to eight times the threads with a
// chain of 8 (SPLIT in dense_mask_draw_kernel): us of a call of 5 recorded sweeps,
// whole / split: L = 64 43 / 36, 512 39 / 34, 1008 (20,160 threads) 53 / 48, 1400
// (38,500) 68 / 63, 1600 (52,000) 75 / 72; but of 10 of L = 1500 (90,000) 80 / 85.
// Not beside a launch that applies masks: there the split costs SM time (300 of L =
// 512 198 / 208).
constexpr long long kSplitThreads = 50000;

// Asynchronous copy of a unit's masks (V words of (r < thr1, r < thr0)) from p
// to shared address dst.
template <int V>
__device__ __forceinline__ void mask_copy(uint32_t dst, const uint64_t* p, const uint64_t* base, uint64_t words,
                                          uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index((uint64_t)(p - base) + (V - 1), words, line)) return;
#else
    (void)base;
    (void)words;
    (void)line;
#endif
    if constexpr (V == 1) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(p) : "memory");
    if constexpr (V == 2) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(p) : "memory");
}
__device__ __forceinline__ void mask_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void mask_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Half-sweep d of a phase, of colour C, on window rows 1 + d .. R - 2 - d: each
// thread updates those of its NS units that lie there.  RECORD counts the
// block's own rows into the count slots `counts`.
template <int V, int C, bool RECORD, int NS>
__device__ __forceinline__ void cl_half_sweep(const uint32_t (&m)[NS][2 * V], uint32_t win0, uint32_t win_bytes,
                                              uint32_t P4, const Slot (&slot)[NS], int d, bool last_lo,
                                              uint32_t live_last, unsigned long long* counts)
{
    uint32_t anti = 0, up = 0;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        if (slot[j].depth >= d) {
            if (RECORD && slot[j].own)
                cl_update<V, C, true>(m[j], win0, win_bytes, P4, slot[j], last_lo, live_last, anti, up);
            else
                cl_update<V, C, false>(m[j], win0, win_bytes, P4, slot[j], last_lo, live_last, anti, up);
        }
    }
    if (RECORD) block_add_counts(counts, anti, up);
}

// V: dense words per unit; NS: units per thread: the block has ceil(units /
// NS) threads, rounded up to whole warps.  DEPTH: half-sweeps a unit's masks
// are copied ahead.  MULTI: several clusters (G > 1), with the
// halo exchange between them; without it the form has no code for that
// exchange.
template <int V, int NS, int DEPTH, bool MULTI>
__global__ void __launch_bounds__(kClThreads, 1)
cluster_sweeps_kernel(ClusterArgs a)
{
    extern __shared__ __align__(16) uint64_t smem[];
    // the next piece's mask draw (launched with programmatic stream
    // serialization) may start now, on the SMs this cluster leaves free
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cg::cluster_group cluster = cg::this_cluster();
    const DenseGeom& g = a.d;
    const int T = blockDim.x;
    const int C = (int)cluster.num_blocks(), b = (int)cluster.block_rank();
    const int k = a.k;
    // the launch's G C blocks own consecutive row bands: block B = gc C + b
    const int G = a.G, gc = (int)blockIdx.x / C, NB = G * C, B = gc * C + b;
    // several clusters: count in (a launch after a piece that gave up does nothing)
    if (__builtin_expect(MULTI && !cl_count_in(a.gate, a.piece), 0)) return;
    // every block of the cluster has started before any block writes into
    // another's shared memory: arrive now, wait just before the first push
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    auto row0 = [&](int blk) { return (int)((long long)blk * g.L / NB); };
    const int r0 = row0(B), r1 = row0(B + 1), S = r1 - r0, R = S + 2 * k;
    const int bp = (b + C - 1) % C, bn = (b + 1) % C;                   // the blocks above and below in the cluster
    // with G > 1 a cluster's first block takes its upper halo from the last
    // block of the cluster above (boundary bd_up, through global memory), its
    // last block the lower halo from the first block of the cluster below
    const bool up_remote = MULTI && b == 0, dn_remote = MULTI && b == C - 1;
    const int bd_up = (gc + G - 1) % G, bd_dn = gc;
    const int top = r0 - k;                                            // global row of window row 0 (mod L)
    const uint32_t P = (uint32_t)g.P;
    const uint64_t n = (uint64_t)a.rmax * P;                            // window words of a colour
    uint32_t* const base32 = reinterpret_cast<uint32_t*>(smem);
    uint32_t* win[2] = {base32, base32 + n};
    const uint32_t smem_sh = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t win_bytes = (uint32_t)n * 4u, P4 = P * 4u;
    const int pairs = g.P / 2;
    const bool last_lo = (g.W & 1) != 0;
    const uint32_t live_last = dense_live(g, g.W - 1);
    const size_t plane = (size_t)g.L * P;                               // one half-sweep's masks
    const uint64_t mask_words = (uint64_t)(2 * a.nsweeps + kClMaskPad) * plane;   // the launch's mask array
    // units: e = t + j T over the rows 1 .. R - 2 of the window
    const int upr = V == 2 ? pairs : g.W;                               // units per row
    Slot slot[NS];
    const uint64_t* msrc[NS];                                           // masks of the next half-sweep to load
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const int e = threadIdx.x + j * T;
        const int lr = 1 + e / upr, w = (e % upr) * V;
        const uint32_t row = (uint32_t)lr * P;
        const bool left0 = ((top + lr) & 1) == 0;
        const uint32_t before = 4u * (row + (uint32_t)(w == 0 ? g.W - 1 : w - 1));
        slot[j].last = w + V >= g.W;
        const uint32_t after = 4u * (row + (uint32_t)(slot[j].last ? 0 : w + V));
        slot[j].depth = lr <= R - 2 ? min(lr - 1, R - 2 - lr) : -1;
        slot[j].at[0] = smem_sh + 4u * (row + (uint32_t)w);
        slot[j].at[1] = slot[j].at[0] + win_bytes;
        slot[j].side[0] = smem_sh + win_bytes + (left0 ? before : after);
        slot[j].side[1] = smem_sh + (left0 ? after : before);
        slot[j].shl = w == 0 ? (uint32_t)(32 - g.lb) : 0u;
        // word 0's bit to bit lb - 1 of the last word where the funnel shift does not put it there
        slot[j].mul = slot[j].last && (g.lb < 32 || (V == 2 && last_lo)) ? 1u << (g.lb - 1) : 0u;
        slot[j].left0 = left0;
        slot[j].own = lr >= k && lr < R - k;
        // units past the window copy row 1's masks and never use them
        msrc[j] = a.masks + (lr <= R - 2 ? (size_t)wrap_index(top + lr, g.L) * P + w
                                         : (size_t)wrap_index(top + 1, g.L) * P);
    }
    // the thread's mask slots: unit j of half-sweep h at slots + j kUnit + (h % DEPTH) kSlab
    constexpr uint32_t kUnit = (uint32_t)kClThreads * 8u * V, kSlab = NS * kUnit;
    static_assert((DEPTH & (DEPTH - 1)) == 0 && (kSlab & (kSlab - 1)) == 0, "the ring's offsets wrap by masking");
    const uint32_t masks_sh = smem_sh + 2u * win_bytes + 64u * (uint32_t)(k * pairs);
    const uint32_t slots = masks_sh + (uint32_t)threadIdx.x * 8u * V;
    uint32_t slab = 0;                                                  // offset of the slab of the next half-sweep to run
    // the masks of the next half-sweep to copy into the slab at `at`, one copy
    // group each (past the end: the planes kClMaskPad adds, never used)
    auto copy_masks = [&](uint32_t at) {
#pragma unroll
        for (int j = 0; j < NS; ++j) {
            mask_copy<V>(slots + at + (uint32_t)j * kUnit, msrc[j], a.masks, mask_words, __LINE__);
            msrc[j] += plane;
        }
        mask_commit();
    };
    // the masks of the half-sweep about to run, and after it the copies that take their place
    auto take_masks = [&](uint32_t (&m)[NS][2 * V]) {
        mask_wait<DEPTH - 1>();
#pragma unroll
        for (int j = 0; j < NS; ++j)
            sh_ld<2 * V>(slots + slab + (uint32_t)j * kUnit, m[j], masks_sh, masks_sh + DEPTH * kSlab, __LINE__);
    };
    auto next_masks = [&]() {
        copy_masks(slab);
        slab = (slab + kSlab) & (DEPTH * kSlab - 1u);
    };
    // halo rows (as 64-bit words): receive slots for the k rows above the
    // block's own (dir 0: the last own rows of the block above) and the k rows
    // below (dir 1), both colours; two sets, used by alternate phases
    const int kP = k * pairs;
    const uint64_t n64 = n / 2;
    uint64_t* const win0 = reinterpret_cast<uint64_t*>(win[0]);        // colour c: + c n64
    uint64_t* recv = smem + n;                                          // [parity][colour][dir] k pairs
    // the global slots between clusters, [boundary][dir][parity][colour]: dir 0
    // carries the last k own rows of cluster bd's last block down to the first
    // block of cluster bd + 1, dir 1 the first k own rows of that block up
    auto xs = [&](int bd, int dir, int par, int c) {
        return a.xbuf + (size_t)(((bd * 2 + dir) * 2 + par) * 2 + c) * kP;
    };
    uint64_t* const up_recv = up_remote ? nullptr : cluster.map_shared_rank(recv, bp);
    uint64_t* const dn_recv = dn_remote ? nullptr : cluster.map_shared_rank(recv, bn);
    // push m (m = 0 before the first phase, m = p + 1 after phase p): a
    // block's first k own rows go to the slots below of the block above, its
    // last k own rows to the slots above of the block below.  Word x: part x /
    // kP = 2 colour + direction.
    auto push = [&](int par, int mth) {
        for (int x = threadIdx.x; x < 4 * kP; x += T) {
            const int part = (x >= kP) + (x >= 2 * kP) + (x >= 3 * kP), c = part >> 1, dir = part & 1;
            const int idx = x - part * kP;
            const uint64_t v =
                word_ld<false>(win0, c * n64 + (uint64_t)(dir ? S : k) * pairs + idx, 2 * n64, __LINE__);
            uint64_t* to;
            if (dir) to = dn_remote ? xs(bd_dn, 0, par, c) : dn_recv + (size_t)((par * 2 + c) * 2 + 0) * kP;
            else to = up_remote ? xs(bd_up, 1, par, c) : up_recv + (size_t)((par * 2 + c) * 2 + 1) * kP;
            word_st(to, idx, v, kP, __LINE__);
        }
        if (up_remote || dn_remote) {
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) {
                if (up_remote) cl_flag_release(a.xflag + bd_up * 2 + 1, a.xseq + mth + 1);
                if (dn_remote) cl_flag_release(a.xflag + bd_dn * 2 + 0, a.xseq + mth + 1);
            }
        }
    };
    // the halos of phase p (push p of the neighbours)
    auto receive = [&](int par, int p) {
        if (up_remote || dn_remote) {
            if (threadIdx.x == 0) {
                if (up_remote) cl_wait_flag(a.xflag + bd_up * 2 + 0, a.xseq + a.xwait + p + 1, a.xerr);
                if (dn_remote) cl_wait_flag(a.xflag + bd_dn * 2 + 1, a.xseq + a.xwait + p + 1, a.xerr);
            }
            __syncthreads();
        }
        for (int x = threadIdx.x; x < 4 * kP; x += T) {
            const int part = (x >= kP) + (x >= 2 * kP) + (x >= 3 * kP), c = part >> 1, dir = part & 1;
            const int idx = x - part * kP;
            uint64_t v;
            if (dir ? dn_remote : up_remote) v = __ldcg((dir ? xs(bd_dn, 1, par, c) : xs(bd_up, 0, par, c)) + idx);
            else v = word_ld<false>(recv, (uint64_t)par * 4 * kP + x, 8 * (uint64_t)kP, __LINE__);
            word_st(win0, c * n64 + (uint64_t)(dir ? k + S : 0) * pairs + idx, v, 2 * n64, __LINE__);
        }
    };
    // own rows of both colours, from the lattice, to window rows k .. k + S - 1
    for (int c = 0; c < 2; ++c)
        for (int e = threadIdx.x; e < S * g.P; e += T) {
            const int r = e / g.P, w = e - r * g.P;
            uint32_t v = 0;
            if (a.dense) v = half_ld(a.dense, ((uint64_t)c * g.L + r0 + r) * P + w, 2 * (uint64_t)g.L * P, __LINE__);
            else if (w < g.W) v = dense_from_packed(a.w[c], (uint64_t)(r0 + r) * a.g.P, a.g, w);
            half_st(win[c], (uint64_t)(k + r) * P + w, v, n, __LINE__);
        }
    __syncthreads();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    push(0, 0);
    for (int h = 0; h < DEPTH; ++h) copy_masks((uint32_t)h * kSlab);
    cluster.sync();          // the first phase's halos have arrived
    // records: sweep j of the launch (1-based) is sweep s0 + j of the call;
    // the next recorded one, rec_j (past nsweeps: none), and its count slot
    int j = 0, rec_j = a.nsweeps + 1;
    unsigned long long* rec_counts = nullptr;
    if (a.every > 0) {
        const int64_t first = (a.s0 / a.every + 1) * a.every;          // first recorded sweep of the call > s0
        if (first - a.s0 <= a.nsweeps) {
            rec_j = (int)(first - a.s0);
            rec_counts = a.counts + ((size_t)(first / a.every - 1) * a.slots + (blockIdx.x & (a.slots - 1))) * 2;
        }
    }
    // d: the half-sweep's number in the phase
    int par = 0, phase = 0, d = 0;
    while (j < a.nsweeps) {
        uint32_t m[NS][2 * V];
        if (d == 0) receive(par, phase);  // into the halo rows (ordered before the updates by the barrier)
        take_masks(m);
        __syncthreads();
        cl_half_sweep<V, 0, false, NS>(m, smem_sh, win_bytes, P4, slot, d, last_lo, live_last, nullptr);
        next_masks();
        take_masks(m);
        __syncthreads();
        if (++j == rec_j) {
            cl_half_sweep<V, 1, true, NS>(m, smem_sh, win_bytes, P4, slot, d + 1, last_lo, live_last, rec_counts);
            rec_counts += 2 * a.slots;
            rec_j = a.every <= a.nsweeps - j ? j + (int)a.every : a.nsweeps + 1;
        } else {
            cl_half_sweep<V, 1, false, NS>(m, smem_sh, win_bytes, P4, slot, d + 1, last_lo, live_last, nullptr);
        }
        next_masks();
        d += 2;
        if (d == k || j == a.nsweeps) {
            d = 0;
            par ^= 1;
            ++phase;
            if (j < a.nsweeps) {
                __syncthreads();     // own rows final for this phase
                push(par, phase);
            }
            // the next phase's halos have arrived; the slots the next pushes write
            // were read at the start of this phase; after the last phase: no block
            // leaves while another may still write its shared memory
            cluster.sync();
        }
    }
    mask_wait<0>();
    // own rows back to the lattice, with several clusters only if every block
    // of the launch was resident (otherwise none writes)
    if (__builtin_expect(MULTI && !cl_decide(a.gate, a.gate_blocks, a.piece), 0)) return;
    if (a.dense) {
        for (int c = 0; c < 2; ++c)
            for (int idx = threadIdx.x; idx < S * (int)P; idx += T)
                half_st(a.dense, ((uint64_t)c * g.L + r0) * P + idx,
                        half_ld(win[c], (uint64_t)k * P + idx, n, __LINE__), 2 * (uint64_t)g.L * P, __LINE__);
        return;
    }
    for (int c = 0; c < 2; ++c)
        for (int e = threadIdx.x; e < S * a.g.W; e += T) {
            const int r = e / a.g.W, w = e - r * a.g.W;
            const int at = kFields * w >> 5;
            const uint64_t o = (uint64_t)(k + r) * P + at;
            const uint32_t d0 = half_ld(win[c], o, n, __LINE__);
            const uint32_t d1 = at + 1 < g.W ? half_ld(win[c], o + 1, n, __LINE__) : 0u;
            word_st(a.w[c], (uint64_t)(r0 + r) * a.g.P + w, packed_from_dense(d0, d1, w), lattice_words(a.g),
                    __LINE__);
        }
}

// The forms of the kernel: one or two dense words per unit, 1 or 2 units per
// thread; one cluster or several.
using ClusterKernel = void (*)(ClusterArgs);
constexpr int kForms = 4;
constexpr int kDepth[kForms] = {8, 8, 8, 4};
static_assert(kClMaskPad >= 8, "the copies run DEPTH half-sweeps ahead");
constexpr ClusterKernel kClusterKernels[2 * kForms] = {
    cluster_sweeps_kernel<1, 1, kDepth[0], false>, cluster_sweeps_kernel<1, 2, kDepth[1], false>,
    cluster_sweeps_kernel<2, 1, kDepth[2], false>, cluster_sweeps_kernel<2, 2, kDepth[3], false>,
    cluster_sweeps_kernel<1, 1, kDepth[0], true>,  cluster_sweeps_kernel<1, 2, kDepth[1], true>,
    cluster_sweeps_kernel<2, 1, kDepth[2], true>,  cluster_sweeps_kernel<2, 2, kDepth[3], true>};

int form(const ClusterPlan& p) { return 2 * (p.v - 1) + p.ns - 1; }

ClusterKernel cluster_kernel(const ClusterPlan& p) { return kClusterKernels[(p.clusters > 1 ? kForms : 0) + form(p)]; }

// Both colour windows (largest share of rows + 2 k rows each), 8 halo receive
// slots of k rows and the threads' mask slots.
size_t cl_smem_bytes(const DenseGeom& d, const ClusterPlan& p)
{
    const int nb = p.clusters * p.blocks, smax = (d.L + nb - 1) / nb;
    return ((size_t)(smax + 2 * p.k) + 4 * (size_t)p.k) * d.P * sizeof(uint64_t) +
           (size_t)kDepth[form(p)] * kClThreads * p.ns * p.v * sizeof(uint64_t);
}

// The blocks of the largest cluster a device runs (0: none), and how many such
// clusters can be resident at once.
struct MaxCluster {
    int size = 0, active = 0;
};

MaxCluster probe_max_cluster()
{
    if (!band_setup()) return {};
    for (ClusterKernel kern : kClusterKernels) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemMax) != cudaSuccess)
            return {};
    }
    for (int c : {16, 8}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = kClSmemMax;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        bool ok = true;
        int active = 1 << 30;
        for (ClusterKernel kern : kClusterKernels) {
            int nc = 0;
            ok = ok && cudaOccupancyMaxActiveClusters(&nc, kern, &cfg) == cudaSuccess && nc >= 1;
            active = std::min(active, nc);
        }
        if (ok) return {c, active};
        cudaGetLastError();
    }
    return {};
}

MaxCluster max_cluster()
{
    static PerDevice<MaxCluster> m;
    return m.get(probe_max_cluster);
}

}  // namespace

int cluster_max_active() { return max_cluster().active; }

// The sides a launch of `blocks` blocks takes (the path's range): at least two
// rows per block (four columns in the column-interleaved layout), and up to
// these.
bool cluster_side(int L, int blocks, bool interleaved)
{
    constexpr struct { int blocks, row, ci; } kMax[] = {
        {8, 1152, 1092},   {16, 1600, 1512},  {24, 1992, 1848},  {32, 2272, 2100},
        {40, 2560, 2352},  {48, 2784, 2688},  {56, 3024, 2856},  {64, 3200, 3024},
        {80, 3600, 3276},  {96, 3936, 3528},  {112, 4256, 3864}};
    if (L < (interleaved ? 4 : 2) * blocks) return false;
    for (const auto& m : kMax)
        if (m.blocks == blocks) return L <= (interleaved ? m.ci : m.row);
    return false;
}

// Cluster size, phase length and units per thread for side L: 16 blocks if the
// device runs such a cluster, else 8; k = the most half-sweeps per phase (even,
// <= kClHalo, <= the fewest rows a block owns) whose window has at most two
// units per thread and fits in shared memory.
bool cluster_plan(int L, bool interleaved, int clusters, ClusterPlan* plan)
{
    const MaxCluster most = max_cluster();
    const int c = most.size;
    if (c == 0 || clusters < 1 || clusters > most.active) return false;
    const int nb = clusters * c, fewest = L / nb;         // blocks of the launch
    if (!cluster_side(L, nb, interleaved)) return false;
    if (clusters == 1 && band_plan(L, c, plan)) return true;
    const DenseGeom d = dense_geom(L);
    for (int kk = std::min(d.W > kClWideWords ? kClHaloWide : kClHalo, fewest) & ~1; kk >= 2; kk -= 2) {
        const long long rows = (L + nb - 1) / nb + 2 * kk - 2;
        const long long words = rows * d.W;
        plan->v = words <= kClOneWord ? 1 : 2;
        const long long units = plan->v == 1 ? words : rows * (d.P / 2);
        plan->ns = (int)((units + kClThreads - 1) / kClThreads);
        if (plan->ns > 2) continue;
        plan->blocks = c;
        plan->k = kk;
        plan->threads = (int)(((units + plan->ns - 1) / plan->ns + 31) / 32 * 32);
        plan->clusters = clusters;
        if (cl_smem_bytes(d, *plan) <= kClSmemMax) return true;
    }
    return false;
}

size_t cl_exchange_words(int L, const ClusterPlan& plan)
{
    return (size_t)plan.clusters * 2 * 2 * 2 * plan.k * (dense_geom(L).P / 2);   // [boundary][dir][parity][colour]
}

unsigned long long cl_exchange_seqs(const ClusterPlan& plan, int nsweeps)
{
    return (unsigned long long)((2 * nsweeps + plan.k - 1) / plan.k) + 1;   // pushes of a launch, + 1
}

size_t cl_mask_bytes_per_sweep(int L) { return 2 * (size_t)L * dense_geom(L).P * sizeof(uint64_t); }

size_t cl_dense_bytes(int L) { return 2 * (size_t)L * dense_geom(L).P * sizeof(uint32_t); }

cudaError_t launch_cl_mask_draw(int L, const SweepArgs& a, uint64_t t0, int nsweeps, uint64_t* masks, bool overlap,
                                cudaStream_t s)
{
    const DenseGeom d = dense_geom(L);
    const Strips st = make_strips(d.P, kDenseStripWords);
    const uint32_t groups = (uint32_t)(L + 3) / 4, items = groups * st.width;
    const bool split = !overlap && (long long)groups * d.P * nsweeps <= kSplitThreads;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = split ? dim3((4 * items + 127) / 128, st.n, 2 * nsweeps) : dim3((items + 127) / 128, st.n, nsweeps);
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    const DenseOut to = {4u * (uint32_t)d.P, (uint32_t)d.P, (uint32_t)L * (uint32_t)d.P};
    const auto draw = split ? (a.rounds == 7 ? dense_mask_draw_kernel<7, 4> : dense_mask_draw_kernel<10, 4>)
                            : (a.rounds == 7 ? dense_mask_draw_kernel<7, 1> : dense_mask_draw_kernel<10, 1>);
    return cudaLaunchKernelEx(&cfg, draw, d, st, a, t0, to, masks);
}

cudaError_t launch_cluster_sweeps(uint64_t* w0, uint64_t* w1, uint32_t* dense, const Geom& g, const SweepArgs& a,
                                  int slots, const ClusterPlan& plan, int nsweeps, const uint64_t* masks, int64_t s0,
                                  int64_t every, const ClusterExchange& x, cudaStream_t s)
{
    const int nb = plan.clusters * plan.blocks;
    ClusterArgs ca;
    ca.w[0] = w0;
    ca.w[1] = w1;
    ca.dense = dense;
    ca.g = g;
    ca.d = dense_geom(g.L);
    ca.k = plan.k;
    ca.nsweeps = nsweeps;
    ca.rmax = (g.L + nb - 1) / nb + 2 * plan.k;
    ca.masks = masks;
    ca.s0 = s0;
    ca.every = every;
    ca.counts = a.counts;
    ca.slots = slots;
    ca.G = plan.clusters;
    ca.xbuf = x.buf;
    ca.xflag = x.flags;
    ca.xseq = x.seq;
    ca.xwait = x.wait_add;
    ca.xerr = x.err;
    ca.gate = x.gate;
    ca.gate_blocks = (unsigned int)(nb) + x.absent;
    ca.piece = x.piece;
    if (plan.clusters > 1 && (!x.buf || !x.flags || !x.err || !x.gate)) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(plan.threads);
    cfg.dynamicSmemBytes = cl_smem_bytes(ca.d, plan);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cluster_kernel(plan), ca);
}

}  // namespace ising
