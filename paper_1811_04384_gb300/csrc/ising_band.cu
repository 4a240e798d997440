// The cluster path on one cluster, rows of 3 to 14 dense words (L up to 896):
// every warp runs its own trapezoid in registers.
//
// What bounds the path at these sides is the latency of a half-sweep, not its
// instructions: with the window in shared memory (cluster_sweeps_kernel) it is
// a mask wait, a block barrier, a shared-memory round trip and a store, 460
// cycles at L = 296.  Here a lane holds a whole row of both colours and a warp
// 32 consecutive rows, of which it owns L / (4 blocks) or so and recomputes k
// on either side (a trapezoid, as the blocks of cluster_sweeps_kernel): the row
// neighbours are two shuffles per word and nothing else is shared for k
// half-sweeps.  Then each lane sends its own row to its block's window and to
// the halos of the blocks above and below (st.async into distributed shared
// memory, counted by the receiving block's barrier), and the warps load their
// 32 rows of the next window.  Two windows are used by alternate phases.  Four
// more warps copy the next phase's masks meanwhile.  A half-sweep of L = 296
// takes 235 cycles with its share of the exchange (96 warp instructions, of which 45 are
// the update).  Measured on GB300, us per call, a record every 10 sweeps, against
// cluster_sweeps_kernel: L = 130 (1000 sweeps) 286 / 535; 296 (1000) 359 / 534;
// 512 (1000) 518 / 640; 704 (1000) 778 / 848; 832 (800) 777 / 798; 896 (600) 628
// / 642; but 960 (500) 566 / 569 and 1088 (500) 702 / 606, so it ends at 14 words.
//
// Tried and slower at L = 296: two rows per lane and k = 18 (no per-lane
// shifts; 470 us against 400 with the same exchange), and a cluster barrier
// after plain stores as the exchange (393 against 357).
#include <cuda_runtime.h>
#include <cooperative_groups.h>

#include <algorithm>
#include <utility>

#include "ising_cluster.cuh"
#include "ising_dense.cuh"
#include "ising_device.cuh"
#include "ising_internal.h"

namespace cg = cooperative_groups;

namespace ising {
namespace {

constexpr int kBandMinWords = 3, kBandMaxWords = 14;
constexpr int kBandWarps = 4;                                 // sweeping warps; as many copy masks
constexpr int kBandThreads = 2 * kBandWarps * 32;

struct BandArgs {
    uint64_t* w[2];             // the lattice's colour arrays (null: `dense`)
    uint32_t* dense;            // or a dense array, [colour][row][word], L x d.P words per colour
    Geom g;
    DenseGeom d;
    int k;                      // half-sweeps per phase = halo rows
    int nsweeps;                // sweeps of this launch
    int rmax;                   // window rows the shared memory holds
    const uint64_t* masks;      // masks[(h * L + i) * d.P + w]: half-sweep h of the launch, row i, word w
    int64_t s0, every;          // as ClusterArgs
    unsigned long long* counts;
    int slots;                  // count slots of a record, a power of two
    uint64_t* t_dev;            // advanced by nsweeps at the end
    unsigned int* err;          // set to 1 when a wait for rows gives up
    int stall;                  // 1: the first wait is for rows that never come (a test hook)
};

// A lane's row of both colours.  The side neighbour of a site of colour C is at
// m - 1 (left) in rows i with i + C even, else at m + 1; the lanes of a warp
// differ in that, so each word is shifted by a lane's own amount between words
// picked by its mask.
template <int W>
struct BandRow {
    uint32_t x[2][W];
    uint32_t left[2];     // all bits: left, for an update of colour 0 and 1
    uint32_t shift[2];    // 31 (left) or 1 (right), for an update of colour 0 and 1
    uint32_t mul[2];      // right: bit lb - 1, where word 0's bit goes across the wrap; left: 0
    uint32_t wrap;        // 32 - lb: the last word's top bit to bit 31

    // The other colour's neighbours of colour C's sites: the rows above (u) and
    // below (d), and to the side (h1; what lands past bit lb - 1 of the last word
    // is not zero).
    template <int C>
    __device__ __forceinline__ void neighbours(uint32_t (&u)[W], uint32_t (&d)[W], uint32_t (&h1)[W]) const
    {
        constexpr int kPick = (kLutA & kLutC) | (kLutB & ~kLutC & 0xff);
        const uint32_t(&h)[W] = x[1 - C];
        uint32_t z[W + 1];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            u[w] = __shfl_up_sync(0xffffffffu, h[w], 1);
            d[w] = __shfl_down_sync(0xffffffffu, h[w], 1);
        }
        z[0] = lop3<kPick>(h[W - 1] << wrap, h[0], left[C]);
#pragma unroll
        for (int w = 1; w < W; ++w) z[w] = lop3<kPick>(h[w - 1], h[w], left[C]);
        z[W] = h[W - 1] & left[C];
#pragma unroll
        for (int w = 0; w < W; ++w) h1[w] = __funnelshift_r(z[w], z[w + 1], shift[C]);
        h1[W - 1] += h[0] * mul[C];
    }

    // One half-sweep of colour C with the row's masks, (r < thr1, r < thr0) of
    // two words per 16 bytes.
    template <int C>
    __device__ __forceinline__ void half_sweep(const uint4 (&m)[(W + 1) / 2])
    {
        uint32_t u[W], d[W], h1[W];
        neighbours<C>(u, d, h1);
#pragma unroll
        for (int w = 0; w < W; ++w)
            x[C][w] = flip_all(x[C][w], u[w], d[w], x[1 - C][w], h1[w], w & 1 ? m[w / 2].z : m[w / 2].x,
                               w & 1 ? m[w / 2].w : m[w / 2].y);
    }

    // The anti-aligned bonds of the row's colour 1 and its up spins.
    __device__ __forceinline__ DenseCount count(uint32_t live_last) const
    {
        uint32_t u[W], d[W], h1[W];
        DenseCount cnt;
        neighbours<1>(u, d, h1);
#pragma unroll
        for (int w = 0; w < W; ++w)
            cnt.add(x[1][w], u[w], d[w], x[0][w], h1[w], w == W - 1 ? live_last : 0xffffffffu);
        return cnt;
    }
};

// A row to a window of a block of the cluster, at byte `off` of its `bytes` at
// `win`; its 16 ceil(W / 4) bytes count towards the block's barrier `bar`.
template <int W>
__device__ __forceinline__ void send(uint32_t win, uint32_t off, uint32_t bytes, uint32_t bar, const uint32_t (&x)[W])
{
#ifdef ISING_CHECKED
    if (!check_index((uint64_t)off + (W + 3) / 4 * 16 - 1, bytes, __LINE__)) return;
#else
    (void)bytes;
#endif
    const uint32_t to = win + off;
#pragma unroll
    for (int w = 0; w < W; w += 4)
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                     ::"r"(to + 4u * w), "r"(x[w]), "r"(w + 1 < W ? x[w + 1 < W ? w + 1 : 0] : 0u),
                     "r"(w + 2 < W ? x[w + 2 < W ? w + 2 : 0] : 0u), "r"(w + 3 < W ? x[w + 3 < W ? w + 3 : 0] : 0u),
                     "r"(bar) : "memory");
}

__device__ __forceinline__ uint32_t in_block(uint32_t addr, int rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}

// Waits for the completion of the barrier's phase of that parity.  The rows
// come from blocks of the same cluster, which run at the same time, so they
// come; all the same the wait gives up after kClWaitNs, sets *err and returns
// false.
__device__ __forceinline__ bool wait_rows(uint32_t bar, uint32_t parity, unsigned int* err)
{
    unsigned long long t0 = 0;
    for (int tries = 0;; ++tries) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
        if (tries < 1000) continue;
        if (*(volatile unsigned int*)err != 0) return false;
        const unsigned long long t = cl_globaltimer();
        if (t0 == 0) t0 = t;
        if (t - t0 > kClWaitNs) {
            *(volatile unsigned int*)err = 1;
            return false;
        }
    }
}

// The end of a launch in which a block gave up, for every thread of every
// block once none sends any more: rows that are still on their way reach the
// windows (a millisecond is a thousand times what one takes) before any block
// leaves.
__device__ __forceinline__ void drain_rows(cg::cluster_group cluster)
{
    constexpr unsigned long long kDrainNs = 1000000;
    if (threadIdx.x == 0) {
        const unsigned long long t0 = cl_globaltimer();
        while (cl_globaltimer() - t0 < kDrainNs) __nanosleep(1000);
    }
    cluster.sync();
}

template <int W>
__global__ void __launch_bounds__(kBandThreads, 1)
band_sweeps_kernel(BandArgs a)
{
    constexpr int CH = (W + 1) / 2;          // 16-byte chunks of a row's masks
    constexpr int MP = CH | 1;               // their pitch in shared memory, odd: no bank conflicts between rows
    constexpr int WV = (W + 3) / 4;          // 16-byte vectors of a window row
    constexpr int WP = 4 * (WV | 1);         // its pitch in words, an odd number of vectors as well
    extern __shared__ __align__(16) uint4 band_smem[];
    // the next piece's mask draw may start now, on the SMs this cluster leaves free
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    cg::cluster_group cluster = cg::this_cluster();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const DenseGeom& g = a.d;
    const int C = (int)cluster.num_blocks(), b = (int)cluster.block_rank(), k = a.k;
    const int bp = (b + C - 1) % C, bn = (b + 1) % C;
    auto row0 = [&](int warp) { return (int)((long long)warp * g.L / (kBandWarps * C)); };
    const int r0 = row0(kBandWarps * b), S = row0(kBandWarps * (b + 1)) - r0, R = S + 2 * k, top = r0 - k;
    const int Sp = row0(kBandWarps * (bp + 1)) - row0(kBandWarps * bp);          // rows of the block above
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint4* const ring = band_smem;                                              // [parity][k][rmax][MP]
    const uint32_t slab = (uint32_t)a.rmax * MP;
    uint32_t* const win = reinterpret_cast<uint32_t*>(band_smem + 2u * k * slab);   // [parity][colour][rmax][WP]
    const uint32_t win_words = 4u * a.rmax * WP;
    uint32_t* const win_up = cluster.map_shared_rank(win, bp);
    uint32_t* const win_dn = cluster.map_shared_rank(win, bn);
    auto at = [&](int par, int c, int r, int w) { return ((uint32_t)(2 * par + c) * a.rmax + r) * WP + w; };
    // word w of own row r (0 .. S - 1) to the windows of parity par that hold the row
    auto put = [&](int par, int c, int r, int w, uint32_t v) {
        half_st(win, at(par, c, k + r, w), v, win_words, __LINE__);
        if (r < k) half_st(win_up, at(par, c, k + Sp + r, w), v, win_words, __LINE__);
        if (r >= S - k) half_st(win_dn, at(par, c, r - (S - k), w), v, win_words, __LINE__);
    };
    const uint32_t win_sh = (uint32_t)__cvta_generic_to_shared(win);
    // arrivals of the windows' rows, one barrier per parity; one that nothing arrives at
    __shared__ uint64_t rows_bar[3];
    __shared__ unsigned int gave_up;         // a block of the cluster gave up
    const uint32_t bar_sh = (uint32_t)__cvta_generic_to_shared(rows_bar);
    const uint32_t window_bytes = (uint32_t)R * 2u * WV * 16u;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_sh) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_sh + 8u) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_sh + 16u) : "memory");
        gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int half_sweeps = 2 * a.nsweeps, phases = (half_sweeps + k - 1) / k;
    // masks of phase p to its ring: a copying warp takes rows of the window, its
    // lanes chunks of rows
    auto copy = [&](int p) {
        constexpr int kRows = 32 / CH;       // rows of a pass
        const int nh = min(k, half_sweeps - p * k), chunk = lane % CH;
        const uint64_t plane = (uint64_t)g.L * g.P;
        if (lane < kRows * CH)
            for (int r = (warp - kBandWarps) * kRows + lane / CH; r < R; r += kBandWarps * kRows) {
                const uint64_t* src = a.masks + ((uint64_t)p * k * g.L + wrap_index(top + r, g.L)) * g.P + 2 * chunk;
                uint32_t dst = (uint32_t)__cvta_generic_to_shared(ring + (p & 1) * k * slab + r * MP + chunk);
#pragma unroll 4
                for (int h = 0; h < nh; ++h, src += plane, dst += slab * 16u) {
#ifdef ISING_CHECKED
                    if (!check_index((uint64_t)(src - a.masks) + 1, (uint64_t)half_sweeps * plane, __LINE__)) continue;
                    if (!check_index((dst - (uint32_t)__cvta_generic_to_shared(ring)) / 16u, 2u * k * slab, __LINE__))
                        continue;
#endif
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
                }
            }
        asm volatile("cp.async.wait_all;" ::: "memory");
    };
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");                 // every block has started
    for (int c = 0; c < 2; ++c)
        for (int e = threadIdx.x; e < S * W; e += kBandThreads) {
            const int r = e / W, w = e - r * W;
            const uint32_t v =
                a.dense ? half_ld(a.dense, ((uint64_t)c * g.L + r0 + r) * g.P + w, 2 * (uint64_t)g.L * g.P, __LINE__)
                        : dense_from_packed(a.w[c], (uint64_t)(r0 + r) * a.g.P, a.g, w);
            put(0, c, r, w, v);
        }
    if (warp >= kBandWarps) copy(0);
    cluster.sync();
    bool stopped = false;                    // uniform over the block: one of its waits gave up
    if (warp >= kBandWarps) {
        for (int p = 0; p < phases && !stopped; ++p) {
            if (p + 1 < phases) copy(p + 1);
            stopped = __syncthreads_or(0) != 0;
        }
    } else {
        // lane l: window row first + l; the own rows at lanes k .. k + own - 1
        const int q = kBandWarps * b + warp, first = row0(q) - r0, own = row0(q + 1) - row0(q);
        const int row = min(first + lane, R - 1);
        const bool is_own = lane >= k && lane < k + own;
        BandRow<W> x;
        const bool even = ((top + row) & 1) == 0;
        x.left[0] = even ? 0xffffffffu : 0u;
        x.left[1] = ~x.left[0];
        x.wrap = (uint32_t)(32 - g.lb);
        x.shift[0] = even ? 31u : 1u;
        x.shift[1] = even ? 1u : 31u;
        x.mul[0] = even ? 0u : 1u << (g.lb - 1);
        x.mul[1] = even ? 1u << (g.lb - 1) : 0u;
        const uint32_t live_last = dense_live(g, W - 1);
        // records: sweep j of the launch (1-based) is sweep s0 + j of the call
        int j = 0, rec_j = a.nsweeps + 1;
        unsigned long long* rec = nullptr;
        if (a.every > 0) {
            const int64_t due = (a.s0 / a.every + 1) * a.every;                 // first recorded sweep of the call > s0
            if (due - a.s0 <= a.nsweeps) {
                rec_j = (int)(due - a.s0);
                rec = a.counts + ((size_t)(due / a.every - 1) * a.slots + (q & (a.slots - 1))) * 2;
            }
        }
        const uint32_t to_own = in_block(win_sh, b), to_up = in_block(win_sh, bp), to_dn = in_block(win_sh, bn);
        const uint32_t bar_own = in_block(bar_sh, b), bar_up = in_block(bar_sh, bp), bar_dn = in_block(bar_sh, bn);
        for (int p = 0; p < phases; ++p) {
            const int nh = min(k, half_sweeps - p * k);
            // window p (the first: by the cluster barrier) and the count of the next one's bytes
            const bool come =
                p == 0 || wait_rows(bar_sh + (a.stall ? 16u : 8u * (p & 1)), (p - 1) >> 1 & 1, a.err);
            if (threadIdx.x == 0 && come && p + 1 < phases)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                             ::"r"(bar_sh + 8u * ((p + 1) & 1)), "r"(window_bytes) : "memory");
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int q = 0; q < WV; ++q) {
                    const uint4 v = vector_ld(win, at(p & 1, c, row, 4 * q), win_words, __LINE__);
                    const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int w = 4 * q; w < min(W, 4 * q + 4); ++w) x.x[c][w] = e[w - 4 * q];
                }
            const uint4* m = ring + (p & 1) * k * slab + row * MP;
            uint4 m0[CH];
            auto load = [&](uint4 (&to)[CH], const uint4* from) {
#ifdef ISING_CHECKED
                if (!check_index((uint64_t)(from - ring) + CH - 1, 2u * k * slab + win_words / 4u, __LINE__)) from = ring;
#endif
#pragma unroll
                for (int c = 0; c < CH; ++c) to[c] = from[c];
            };
            load(m0, m);
            for (int h = 0; h < nh; h += 2, m += 2 * slab) {
                uint4 m1[CH];
                load(m1, m + slab);
                x.template half_sweep<0>(m0);
                load(m0, m + 2 * slab);          // past the phase's end: the next ring or the windows, never used
                x.template half_sweep<1>(m1);
                if (++j == rec_j) {
                    const DenseCount cnt = x.count(live_last);
                    // both sums in one reduction: at most 28 own rows of 32 W sites of a colour
                    static_assert(28 * kBandMaxWords * 32 * 4 < 1 << 16, "16 bits each");
                    const uint32_t sum = __reduce_add_sync(0xffffffffu, is_own ? cnt.anti() | cnt.up() << 16 : 0u);
                    if (lane == 0) {
                        atomicAdd(rec, (unsigned long long)(sum & 0xffffu));
                        atomicAdd(rec + 1, (unsigned long long)(sum >> 16));
                    }
                    rec += 2 * a.slots;
                    rec_j = a.every <= a.nsweeps - j ? j + (int)a.every : a.nsweeps + 1;
                }
            }
            // All warps have loaded their rows of window p, so the neighbours may write
            // the window after next (they cannot be there before this block's rows of
            // the next one reach them), the masks of phase p + 1 are in the ring, and
            // those of phase p are no longer needed.  A block that gave up sends
            // nothing more.
            stopped = __syncthreads_or(!come) != 0;
            if (stopped) break;
            if (is_own) {
                // row `row` of the window; row + Sp of the block's above, row - S of the block's below
                const int r = row - k, to = (p + 1) & 1;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const uint32_t o = 4u * at(to, c, row, 0), bar = 8u * to;
                    if (p + 1 < phases) {
                        send(to_own, o, 4u * win_words, bar_own + bar, x.x[c]);
                        if (r < k) send(to_up, o + 4u * WP * Sp, 4u * win_words, bar_up + bar, x.x[c]);
                        if (r >= S - k) send(to_dn, o - 4u * WP * S, 4u * win_words, bar_dn + bar, x.x[c]);
                    } else {
#pragma unroll
                        for (int w = 0; w < W; ++w) half_st(win, at(to, c, row, w), x.x[c][w], win_words, __LINE__);
                    }
                }
            }
        }
    }
    // the own rows are in the window; no block leaves while another may still use its barriers
    if (stopped && threadIdx.x < C) *cluster.map_shared_rank(&gave_up, threadIdx.x) = 1;
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(a.t_dev), (unsigned long long)a.nsweeps);
    if (gave_up) {                           // nobody writes back: the launch leaves the lattice as it was
        drain_rows(cluster);
        return;
    }
    const int par = phases & 1;
    if (a.dense) {
        for (int c = 0; c < 2; ++c)
            for (int e = threadIdx.x; e < S * W; e += kBandThreads) {
                const int r = e / W, w = e - r * W;
                half_st(a.dense, ((uint64_t)c * g.L + r0 + r) * g.P + w,
                        half_ld(win, at(par, c, k + r, w), win_words, __LINE__), 2 * (uint64_t)g.L * g.P, __LINE__);
            }
        return;
    }
    for (int c = 0; c < 2; ++c)
        for (int e = threadIdx.x; e < S * a.g.W; e += kBandThreads) {
            const int r = e / a.g.W, w = e - r * a.g.W, d = kFields * w >> 5;
            const uint32_t d0 = half_ld(win, at(par, c, k + r, d), win_words, __LINE__);
            const uint32_t d1 = d + 1 < W ? half_ld(win, at(par, c, k + r, d + 1), win_words, __LINE__) : 0u;
            word_st(a.w[c], (uint64_t)(r0 + r) * a.g.P + w, packed_from_dense(d0, d1, w), lattice_words(a.g), __LINE__);
        }
}

using BandKernel = void (*)(BandArgs);
template <int... I>
constexpr BandKernel band_kernel_of(int W, std::integer_sequence<int, I...>)
{
    constexpr BandKernel kernels[] = {band_sweeps_kernel<kBandMinWords + I>...};
    return kernels[W - kBandMinWords];
}
BandKernel band_kernel(int W)
{
    return band_kernel_of(W, std::make_integer_sequence<int, kBandMaxWords - kBandMinWords + 1>());
}

size_t band_smem_bytes(int L, const ClusterPlan& p)
{
    const DenseGeom d = dense_geom(L);
    const size_t rmax = (size_t)(L + p.blocks - 1) / p.blocks + 2 * p.k + 1;
    return 2 * p.k * rmax * ((d.W + 1) / 2 | 1) * 16 + 4 * rmax * 16 * ((d.W + 3) / 4 | 1);
}

}  // namespace

// k: the most half-sweeps a warp's 32 rows allow (its own rows and a halo on
// either side), the halo within the neighbouring blocks.
bool band_plan(int L, int blocks, ClusterPlan* plan)
{
    const int W = dense_geom(L).W, warps = kBandWarps * blocks, own = (L + warps - 1) / warps;
    if (W < kBandMinWords || W > kBandMaxWords) return false;
    plan->blocks = blocks;
    plan->clusters = 1;
    plan->v = 0;
    plan->threads = kBandThreads;
    for (plan->k = std::min((32 - own) / 2, L / blocks) & ~1; plan->k >= 2; plan->k -= 2)
        if (band_smem_bytes(L, *plan) <= kClSmemMax) return true;
    return false;
}

bool band_setup()
{
    for (int W = kBandMinWords; W <= kBandMaxWords; ++W) {
        if (cudaFuncSetAttribute(band_kernel(W), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaFuncSetAttribute(band_kernel(W), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemMax) !=
                cudaSuccess)
            return false;
    }
    return true;
}

cudaError_t launch_band_sweeps(uint64_t* w0, uint64_t* w1, uint32_t* dense, const Geom& g,
                               unsigned long long* counts, int slots, const ClusterPlan& plan, int nsweeps,
                               const uint64_t* masks, int64_t s0, int64_t every, uint64_t* t_dev,
                               unsigned int* err, bool stall, cudaStream_t s)
{
    BandArgs a;
    a.w[0] = w0;
    a.w[1] = w1;
    a.dense = dense;
    a.g = g;
    a.d = dense_geom(g.L);
    a.k = plan.k;
    a.nsweeps = nsweeps;
    a.rmax = (g.L + plan.blocks - 1) / plan.blocks + 2 * plan.k + 1;
    a.masks = masks;
    a.s0 = s0;
    a.every = every;
    a.counts = counts;
    a.slots = slots;
    a.t_dev = t_dev;
    a.err = err;
    a.stall = stall;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.blocks);
    cfg.blockDim = dim3(kBandThreads);
    cfg.dynamicSmemBytes = kClSmemMax;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = plan.blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, band_kernel(a.d.W), a);
}

}  // namespace ising
