// The on-chip path of small lattices (L <= 128): one warp holds the whole
// lattice in registers, one bit per spin (ising_dense.cuh), and runs all sweeps
// of a call from accept masks drawn beforehand on all SMs.
//
// What bounds it: the chain of dependent half-sweeps.  A block with the
// lattice in shared memory paid a block barrier, six shared-memory loads and
// the index arithmetic of a packed word per half-sweep: 0.42 us per recorded
// sweep at L = 64, 0.92 at L = 128.  In one warp a half-sweep is two shuffles
// (the rows above and below a lane's own), seven three-input operations per 32
// sites and no barrier.  Measured on GB300: a sweep without a record 69 ns at L
// = 64 and 193 at L = 128 (there the warp's issue slots bind), 1000 recorded
// sweeps of L = 64 in 84 us, against 418 in shared memory, 271 with one warp that
// also copied the masks and counted the records, 159 with three helpers that did
// both, and 218 ns a sweep at L = 128 with the copying warp on the sweeping warp's
// scheduler.
#include <cuda_runtime.h>

#include <algorithm>

#include "ising_dense.cuh"
#include "ising_device.cuh"
#include "ising_internal.h"

namespace ising {
namespace {

// Warp 0 sweeps, warp 4 leaves that scheduler to it, warp 5 copies masks, the
// others count records.
constexpr int kWarpThreads = 256, kIdle = 4, kCopier = 5, kCounters = kWarpThreads / 32 - 3;

// Word rows without a pad: one word, or two.
DenseGeom warp_geom(int L)
{
    DenseGeom d = dense_geom(L);
    d.P = d.W;
    return d;
}

// Lane l holds rows RPL l .. RPL l + RPL - 1 (RPL even, so a row's parity is
// its register's) of W dense words of both colours; lanes past the last row
// run along and are never read.  TWO: L % 4 == 2 with RPL = 4, so the last lane
// holds two rows.
template <int W, int RPL, bool TWO>
struct WarpLattice {
    uint32_t x[2][RPL][W];
    int prev, next;       // lanes of the rows above and below (periodic)
    bool tail;            // the lane of two rows
    uint32_t lsh, mul;    // lb - 1 and 2^(lb - 1): the row's wrap

    // The other colour's horizontal neighbours at m - 1 (LEFT) or m + 1 of a
    // row; what lands past bit lb - 1 meets masks that are zero.
    template <bool LEFT>
    __device__ __forceinline__ void side(const uint32_t (&h)[W], uint32_t (&y)[W]) const
    {
        if constexpr (W == 1) {
            y[0] = LEFT ? h[0] * 2u + (h[0] >> lsh) : h[0] * mul + (h[0] >> 1);
        } else {
            y[0] = LEFT ? h[0] * 2u + (h[1] >> lsh) : __funnelshift_r(h[0], h[1], 1);
            y[1] = LEFT ? __funnelshift_l(h[0], h[1], 1) : h[0] * mul + (h[1] >> 1);
        }
    }

    // Row neighbours of colour C's rows in the other colour: the lanes' edge
    // rows, and row r's inside the lane.
    template <int C>
    __device__ __forceinline__ void edges(uint32_t (&above)[W], uint32_t (&below)[W]) const
    {
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint32_t bottom = TWO && tail ? x[1 - C][1][w] : x[1 - C][RPL - 1][w];
            above[w] = __shfl_sync(0xffffffffu, bottom, prev);
            below[w] = __shfl_sync(0xffffffffu, x[1 - C][0][w], next);
        }
    }

    template <int C>
    __device__ __forceinline__ void vertical(int r, int w, const uint32_t (&above)[W], const uint32_t (&below)[W],
                                             uint32_t& u, uint32_t& d) const
    {
        u = r == 0 ? above[w] : x[1 - C][r > 0 ? r - 1 : 0][w];
        d = r == RPL - 1 ? below[w] : x[1 - C][r < RPL - 1 ? r + 1 : r][w];
        if (TWO && r == 1) d = tail ? below[w] : d;
    }

    // One half-sweep of colour C with masks m[row][word] = (r < thr1, r < thr0).
    template <int C>
    __device__ __forceinline__ void half_sweep(const uint32_t (&m)[RPL][2 * W])
    {
        uint32_t above[W], below[W];
        edges<C>(above, below);
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            uint32_t h1[W];
            if (((r + C) & 1) == 0) side<true>(x[1 - C][r], h1);
            else side<false>(x[1 - C][r], h1);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                uint32_t u, d;
                vertical<C>(r, w, above, below, u, d);
                x[C][r][w] = flip_all(x[C][r][w], u, d, x[1 - C][r][w], h1[w], m[r][2 * w], m[r][2 * w + 1]);
            }
        }
    }

    // The anti-aligned bonds of colour 1's rows and the up spins of both
    // colours (live bits only) of a lane with rows.
    __device__ __forceinline__ DenseCount count(const uint32_t (&live)[W]) const
    {
        uint32_t above[W], below[W];
        DenseCount cnt;
        edges<1>(above, below);
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            uint32_t h1[W];
            if ((r & 1) == 1) side<true>(x[0][r], h1);
            else side<false>(x[0][r], h1);
            if (TWO && r >= 2 && tail) continue;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                uint32_t u, d;
                vertical<1>(r, w, above, below, u, d);
                cnt.add(x[1][r][w], u, d, x[0][r][w], h1[w], live[w]);
            }
        }
        return cnt;
    }
};

// Sweeps s_base + 1 .. s_base + n of a run with the masks of
// dense_mask_draw_kernel as launch_warp_mask_draw lays them out: rows of 16
// bytes per lane, 2 C of them a sweep.  Warp 0 sweeps; warp kCopier copies the masks
// into a ring of STAGES stages of K sweeps, and the other warps (on the other
// schedulers) count the records, (E, M) of the run's sweeps s with s % every == 0 to
// records[2 (s / every - 1)], from the states that warp 0 leaves in shared
// memory.  One barrier per stage.  At the end *t_dev += n.  Launched
// programmatically behind the mask draw, which no kernel overlaps, so the
// lattice is there before the wait.
template <int W, int RPL, bool TWO, int K, int STAGES>
__global__ void __launch_bounds__(kWarpThreads)
warp_sweeps_kernel(uint64_t* __restrict__ w0, uint64_t* __restrict__ w1, Geom g, DenseGeom d,
                   const uint4* __restrict__ masks, int s_base, int n, int every, long long* records,
                   uint64_t* t_dev)
{
    constexpr int C = W == 1 ? 1 : RPL;          // 16-byte mask chunks of a lane per half-sweep; also of a state
    static_assert(RPL * W == 2 * C, "a chunk holds the masks of two words");
    __shared__ uint4 ring[STAGES][2 * K * C][32];
    __shared__ uint4 state[2][K][C][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, last = (g.L + RPL - 1) / RPL - 1;
    const int prev = lane == 0 ? last : lane - 1, next = lane == last ? 0 : lane + 1;
    const int stages = (n + K - 1) / K;
    uint32_t live[W];
#pragma unroll
    for (int w = 0; w < W; ++w) live[w] = dense_live(d, w);
    WarpLattice<W, RPL, TWO> lat;
    lat.prev = prev;
    lat.next = next;
    lat.tail = TWO && lane == last;
    lat.lsh = (uint32_t)(d.lb - 1);
    lat.mul = 1u << (d.lb - 1);
    if (warp != 0) {
        const long long N = (long long)g.L * g.L;
        auto copy = [&](int stage) {
            if (stage < stages && lane <= last) {
                const int slot = stage % STAGES, rows = 2 * C * min(K, n - stage * K);
                const uint64_t nl = last + 1u, base = (uint64_t)stage * (2 * K * C) * nl + lane;
                for (int r = 0; r < rows; ++r) {
#ifdef ISING_CHECKED
                    if (!check_index(base + r * nl, (uint64_t)n * (2 * C) * nl, __LINE__)) continue;
#endif
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                                 ::"r"((uint32_t)__cvta_generic_to_shared(&ring[slot][r][lane])),
                                   "l"(masks + base + r * nl) : "memory");
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // counter h takes every kCounters-th record of the run: the next one is
        // after sweep `due` of this launch
        const int h = warp < kIdle ? warp - 1 : warp - 3;
        const long long r0 = s_base / every + h;
        long long due = (r0 + 1) * every - s_base;
        long long* rec = records + 2 * r0;
        auto count = [&](int stage) {
            for (; due <= min((stage + 1) * K, n); due += (long long)kCounters * every, rec += 2 * kCounters) {
                const int q = (int)due - 1 - stage * K;
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const uint4 v = state[stage & 1][q][c][lane];
                    if constexpr (W == 1) {
                        lat.x[0][0][0] = v.x; lat.x[0][1][0] = v.y; lat.x[1][0][0] = v.z; lat.x[1][1][0] = v.w;
                    } else {
                        lat.x[0][c][0] = v.x; lat.x[0][c][W - 1] = v.y; lat.x[1][c][0] = v.z; lat.x[1][c][W - 1] = v.w;
                    }
                }
                const DenseCount cnt = lat.count(live);
                // both sums in one reduction: at most 2 L^2 <= 2^15 bonds and 2^14 spins
                const uint32_t sum = __reduce_add_sync(0xffffffffu, lane <= last ? cnt.anti() | cnt.up() << 16 : 0u);
                if (lane == 0) {
                    rec[0] = 2 * (long long)(sum & 0xffffu) - 2 * N;
                    rec[1] = 2 * (long long)(sum >> 16) - N;
                }
            }
        };
        pdl_wait();                                 // the masks are drawn
        if (warp == kCopier) {
            for (int k = 0; k < STAGES - 1; ++k) copy(k);
            asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        }
        __syncthreads();
        for (int k = 0; k < stages; ++k) {
            if (warp == kCopier) {
                copy(k + STAGES - 1);
                asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
            } else if (warp != kIdle && k > 0) {
                count(k - 1);
            }
            __syncthreads();
        }
        if (warp != kCopier && warp != kIdle) count(stages - 1);
        return;
    }

    const int nrows = lane > last ? 0 : min(RPL, g.L - RPL * lane);
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < RPL; ++r)
#pragma unroll
            for (int w = 0; w < W; ++w)
                lat.x[c][r][w] =
                    r < nrows ? dense_from_packed(c ? w1 : w0, (uint64_t)(RPL * lane + r) * g.P, g, w) : 0u;
    pdl_wait();
    __syncthreads();
    int slot = 0;
    for (int k = 0; k < stages; ++k) {
        const int cnt = min(K, n - k * K);
        uint32_t m[2][RPL][2 * W];
        auto take = [&](int h) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const uint4 v = ring[slot][h * C + c][lane];
                uint32_t(&to)[RPL][2 * W] = m[h & 1];
                if constexpr (W == 1) {
                    to[0][0] = v.x; to[0][1] = v.y; to[1][0] = v.z; to[1][1] = v.w;
                } else {
                    to[c][0] = v.x; to[c][1] = v.y; to[c][2 * W - 2] = v.z; to[c][2 * W - 1] = v.w;
                }
            }
        };
        take(0);
#pragma unroll
        for (int q = 0; q < K; ++q) {
            if (q >= cnt) break;
            take(2 * q + 1);
            lat.template half_sweep<0>(m[0]);
            if (q + 1 < K) take(2 * q + 2);
            lat.template half_sweep<1>(m[1]);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if constexpr (W == 1)
                    state[k & 1][q][c][lane] = make_uint4(lat.x[0][0][0], lat.x[0][1][0], lat.x[1][0][0], lat.x[1][1][0]);
                else
                    state[k & 1][q][c][lane] =
                        make_uint4(lat.x[0][c][0], lat.x[0][c][W - 1], lat.x[1][c][0], lat.x[1][c][W - 1]);
            }
        }
        slot = slot + 1 == STAGES ? 0 : slot + 1;
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            if (r >= nrows) continue;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                if (w >= g.W) continue;
                const int at = kFields * w >> 5;                          // 0, 0, 1, 1 (W = 1: fields past 31 are dead)
                const uint32_t d0 = at < W ? lat.x[c][r][at < W ? at : 0] : 0u;
                const uint32_t d1 = at + 1 < W ? lat.x[c][r][at + 1 < W ? at + 1 : 0] : 0u;
                word_st(c ? w1 : w0, (uint64_t)(RPL * lane + r) * g.P + w, packed_from_dense(d0, d1, w),
                        lattice_words(g), __LINE__);
            }
        }
    if (lane == 0) atomicAdd(reinterpret_cast<unsigned long long*>(t_dev), (unsigned long long)n);
}

}  // namespace

size_t warp_mask_bytes_per_sweep(int L)
{
    const DenseGeom d = warp_geom(L);
    return 2 * (size_t)((L + 3) / 4 * 4) * d.P * sizeof(uint64_t);
}

cudaError_t launch_warp_mask_draw(int L, const SweepArgs& a, uint64_t t0, int nsweeps, uint64_t* masks,
                                  cudaStream_t s)
{
    const DenseGeom d = warp_geom(L);
    const Strips st = make_strips(d.P, kDenseStripWords);
    const uint32_t G = (uint32_t)(L + 3) / 4, threads = 4 * G * d.P;
    const uint32_t block = std::min((threads + 31) / 32 * 32, 128u);
    const DenseOut out = d.W == 1 ? DenseOut{4, 1, (uint32_t)L} : DenseOut{2, 2 * G, 8 * G};
    const dim3 grid((threads + block - 1) / block, 1, 2 * nsweeps);
    if (a.rounds == 7)
        dense_mask_draw_kernel<7, 4><<<grid, block, 0, s>>>(d, st, a, t0, out, masks);
    else
        dense_mask_draw_kernel<10, 4><<<grid, block, 0, s>>>(d, st, a, t0, out, masks);
    return cudaGetLastError();
}

cudaError_t launch_warp_sweeps(uint64_t* w0, uint64_t* w1, const Geom& g, const uint64_t* masks, int s_base, int n,
                               int every, long long* rec, uint64_t* t_dev, cudaStream_t s)
{
    const DenseGeom d = warp_geom(g.L);
    const dim3 one(1), block(kWarpThreads);
    const uint4* m = reinterpret_cast<const uint4*>(masks);
    if (d.W == 1)
        launch_pdl(warp_sweeps_kernel<1, 2, false, 8, 3>, one, block, s, w0, w1, g, d, m, s_base, n, every, rec, t_dev);
    else if (g.L % 4 == 0)
        launch_pdl(warp_sweeps_kernel<2, 4, false, 2, 5>, one, block, s, w0, w1, g, d, m, s_base, n, every, rec,
                   t_dev);
    else
        launch_pdl(warp_sweeps_kernel<2, 4, true, 2, 5>, one, block, s, w0, w1, g, d, m, s_base, n, every, rec,
                   t_dev);
    return cudaGetLastError();
}

}  // namespace ising
