// The on-chip path of small lattices (L <= 128): one warp holds the whole
// lattice in registers, one bit per spin (ising_dense.cuh), and runs all sweeps
// of a call from accept masks drawn beforehand on all SMs.
//
// What bounds it: the chain of dependent half-sweeps.  A block with the
// lattice in shared memory paid a block barrier, six shared-memory loads and
// the index arithmetic of a packed word per half-sweep: 0.42 us per recorded
// sweep at L = 64, 0.92 at L = 128.  In one warp a half-sweep is two shuffles
// (the rows above and below a lane's own), seven three-input operations per 32
// sites and no barrier.
#include <cuda_runtime.h>

#include "ising_dense.cuh"
#include "ising_device.cuh"
#include "ising_internal.h"

namespace ising {
namespace {

constexpr int kWarpDepth = 8;       // half-sweeps a row's masks are copied ahead
static_assert(kClMaskPad >= kWarpDepth, "the copies run that far past the last half-sweep");

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

    // One half-sweep of colour C with masks m[row][word] = (r < thr1, r < thr0).
    // RECORD: the anti-aligned bonds of the updated rows and the up spins of
    // both colours (live bits only), below nrows of the lane's rows.
    template <int C, bool RECORD>
    __device__ __forceinline__ void half_sweep(const uint32_t (&m)[RPL][2 * W], int nrows, const uint32_t (&live)[W],
                                               uint32_t& anti, uint32_t& up)
    {
        uint32_t above[W], below[W];
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const uint32_t bottom = TWO && tail ? x[1 - C][1][w] : x[1 - C][RPL - 1][w];
            above[w] = __shfl_sync(0xffffffffu, bottom, prev);
            below[w] = __shfl_sync(0xffffffffu, x[1 - C][0][w], next);
        }
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            uint32_t h1[W];
            if (((r + C) & 1) == 0) side<true>(x[1 - C][r], h1);
            else side<false>(x[1 - C][r], h1);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const uint32_t u = r == 0 ? above[w] : x[1 - C][r > 0 ? r - 1 : 0][w];
                uint32_t d = r == RPL - 1 ? below[w] : x[1 - C][r < RPL - 1 ? r + 1 : r][w];
                if (TWO && r == 1) d = tail ? below[w] : d;
                const uint32_t h0 = x[1 - C][r][w];
                const uint32_t s = flip_all(x[C][r][w], u, d, h0, h1[w], m[r][2 * w], m[r][2 * w + 1]);
                x[C][r][w] = s;
                if (RECORD && r < nrows) {
                    anti += __popc(s ^ u) + __popc(s ^ d) + __popc(s ^ h0) + __popc((s ^ h1[w]) & live[w]);
                    up += __popc(s) + __popc(h0);
                }
            }
        }
    }
};

// Sweeps s_base + 1 .. s_base + n of a run with the masks of
// dense_mask_draw_kernel (P = 2: 16 bytes a row), a record after each of the
// run's sweeps s with s % every == 0 at records[2 (s / every - 1)] as (E, M);
// then *t_dev = t_end.  Launched programmatically behind the mask draw, which
// no kernel overlaps, so the lattice is there before the wait.
template <int W, int RPL, bool TWO>
__global__ void __launch_bounds__(32)
warp_sweeps_kernel(uint64_t* __restrict__ w0, uint64_t* __restrict__ w1, Geom g, DenseGeom d,
                   const uint64_t* __restrict__ masks, int s_base, int n, int every, long long* records,
                   uint64_t* t_dev, uint64_t t_end)
{
    __shared__ __align__(16) uint4 ring[kWarpDepth][RPL][32];
    const int lane = threadIdx.x, last = (g.L + RPL - 1) / RPL - 1;
    WarpLattice<W, RPL, TWO> lat;
    lat.prev = lane == 0 ? last : lane - 1;
    lat.next = lane == last ? 0 : lane + 1;
    lat.tail = TWO && lane == last;
    lat.lsh = (uint32_t)(d.lb - 1);
    lat.mul = 1u << (d.lb - 1);
    const int nrows = lane > last ? 0 : min(RPL, g.L - RPL * lane);
    uint32_t live[W];
#pragma unroll
    for (int w = 0; w < W; ++w) live[w] = dense_live(d, w);
    // masks: the lane's rows (row 0's for rows it does not have, never used)
    const uint64_t plane = (uint64_t)g.L * d.P, mask_words = (2 * (uint64_t)n + kClMaskPad) * plane;
    const uint32_t ring_sh = (uint32_t)__cvta_generic_to_shared(&ring[0][0][lane]);
    constexpr uint32_t kRow = 32 * sizeof(uint4), kSlab = RPL * kRow;
    const uint64_t* src[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) src[r] = masks + (r < nrows ? (uint64_t)(RPL * lane + r) * d.P : 0);
    auto copy = [&](int slab) {
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
#ifdef ISING_CHECKED
            if (check_index((uint64_t)(src[r] - masks) + 1, mask_words, __LINE__))
#endif
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring_sh + (uint32_t)slab * kSlab + r * kRow),
                         "l"(src[r]) : "memory");
            src[r] += plane;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto take = [&](int slab, uint32_t (&m)[RPL][2 * W]) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kWarpDepth - 1) : "memory");
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const uint32_t at = ring_sh + (uint32_t)slab * kSlab + r * kRow;
            if constexpr (W == 1)
                asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(m[r][0]), "=r"(m[r][1]) : "r"(at));
            else
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(m[r][0]), "=r"(m[r][1]), "=r"(m[r][2]), "=r"(m[r][3]) : "r"(at));
        }
    };
    (void)mask_words;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int r = 0; r < RPL; ++r)
#pragma unroll
            for (int w = 0; w < W; ++w)
                lat.x[c][r][w] =
                    r < nrows ? dense_from_packed(c ? w1 : w0, (uint64_t)(RPL * lane + r) * g.P, g, w) : 0u;
    pdl_wait();                                     // the masks are drawn
#pragma unroll
    for (int h = 0; h < kWarpDepth; ++h) copy(h);
    const long long N = (long long)g.L * g.L;
    int next_rec = every - s_base % every;          // the next recorded sweep of this launch
    long long* rec = records + 2 * (s_base / every);
    for (int s0 = 0; s0 < n; s0 += kWarpDepth / 2) {
#pragma unroll
        for (int q = 0; q < kWarpDepth / 2; ++q) {
            const int s = s0 + q + 1;
            if (s > n) break;
            uint32_t m[RPL][2 * W], anti = 0, up = 0;
            take(2 * q, m);
            lat.template half_sweep<0, false>(m, nrows, live, anti, up);
            copy(2 * q);
            take(2 * q + 1, m);
            if (s == next_rec) {
                lat.template half_sweep<1, true>(m, nrows, live, anti, up);
                // both sums in one reduction: anti <= 2 L^2 <= 2^15 and up <= 2^14
                const uint32_t sum = __reduce_add_sync(0xffffffffu, anti | up << 16);
                if (lane == 0) {
                    rec[0] = 2 * (long long)(sum & 0xffffu) - 2 * N;
                    rec[1] = 2 * (long long)(sum >> 16) - N;
                }
                rec += 2;
                next_rec = every <= n - s ? s + every : n + 1;
            } else {
                lat.template half_sweep<1, false>(m, nrows, live, anti, up);
            }
            copy(2 * q + 1);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
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
    if (lane == 0) *t_dev = t_end;
}

}  // namespace

cudaError_t launch_warp_sweeps(uint64_t* w0, uint64_t* w1, const Geom& g, const uint64_t* masks, int s_base, int n,
                               int every, long long* rec, uint64_t* t_dev, uint64_t t_end, cudaStream_t s)
{
    const DenseGeom d = dense_geom(g.L);
    const dim3 one(1), block(32);
    if (d.W == 1)
        launch_pdl(warp_sweeps_kernel<1, 2, false>, one, block, s, w0, w1, g, d, masks, s_base, n, every, rec, t_dev,
                   t_end);
    else if (g.L % 4 == 0)
        launch_pdl(warp_sweeps_kernel<2, 4, false>, one, block, s, w0, w1, g, d, masks, s_base, n, every, rec, t_dev,
                   t_end);
    else
        launch_pdl(warp_sweeps_kernel<2, 4, true>, one, block, s, w0, w1, g, d, masks, s_base, n, every, rec, t_dev,
                   t_end);
    return cudaGetLastError();
}

}  // namespace ising
