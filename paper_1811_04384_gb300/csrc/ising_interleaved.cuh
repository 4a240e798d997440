// Device helpers of the paper's column-interleaved layout (Sec. 3, Fig. 1-2),
// shared by its kernels: the field rotations across the top and bottom word
// rows, and the accept masks of four words from the sites' own Philox draws.
#pragma once
#include <cstdint>

#include "ising_device.cuh"
#include "philox.cuh"

namespace ising {
namespace {

constexpr uint64_t kAllFields = 0x1249249249249249ull;   // bit 3k, k = 0..20

__device__ __forceinline__ uint64_t rotate_up(uint64_t s)    // field k <- field k - 1 (periodic)
{
    return ((s << 3) | (s >> 60)) & kAllFields;
}

__device__ __forceinline__ uint64_t rotate_down(uint64_t s)  // field k <- field k + 1 (periodic)
{
    return ((s >> 3) | (s << 60)) & kAllFields;
}

// Accept masks of the words of column pair m in word rows 4q .. 4q + 3, colour
// C, at sweep t: Philox call k (counter (q + kN/4, m, t, C)) gives the draws
// of field k of the four words, in ItemMasks' form.  Along the 21 calls the
// column stays and the row group changes, so the first product (column and
// sweep) is the thread's own, once, and what depends on the row group alone
// is shared by all columns of a block (ci_row_keys): 15 products per call, as
// in the row-packed layout, where each call's own row key made them 19.
constexpr int kCiBlockX = 32, kCiBlockY = 4;      // column pairs x word row groups of a block of 128

// All threads of a block of kCiBlockX x kCiBlockY (1-D thread index): the row
// keys of row groups q0 .. q0 + GROUPS - 1.
template <int GROUPS>
__device__ __forceinline__ void ci_row_keys(uint4* tab, int N, int q0, uint64_t t, int C, const SweepArgs& a)
{
    static_assert(kCiBlockX * kCiBlockY >= GROUPS * kFields, "one entry per thread");
    const int e = (int)threadIdx.x;
    if (e < GROUPS * kFields) {
        const int y = e / kFields, k = e - y * kFields;
        const PhiloxRowKey pk =
            philox_row_key((uint32_t)(q0 + y + k * (N / 4)), (uint32_t)t, counter_high(t, C), a.rk);
        tab[e] = make_uint4(pk.y3k, pk.z1k, pk.hiC, pk.v3);
    }
    __syncthreads();
}

struct CiCalls {
    const uint4* keys;        // the thread's row group in the table
    uint32_t hi, lo;          // the column's first product
    template <int ROUNDS>
    __device__ __forceinline__ void call(int k, const PhiloxKeys& rk, uint32_t rnd[4]) const
    {
        const uint4 e = keys[k];
        const PhiloxRowKey pk = {0, e.x, e.y, e.z, e.w};
        philox_row_tail<ROUNDS>(pk, rk, hi, lo, rnd);
    }
};

// `tab` from ci_row_keys for the thread's t and C; y the row group in it.
template <int ROUNDS>
__device__ __forceinline__ void ci_masks(const uint4* tab, int y, int m, uint64_t t, const SweepArgs& a,
                                         ItemMasks& acc)
{
    CiCalls calls;
    calls.keys = tab + y * kFields;
    mul_hilo(kPhiloxM0, philox_first_key((uint32_t)t, a.rk) ^ (uint32_t)m, calls.hi, calls.lo);
    draw_fields<ROUNDS>(calls, a.rk, a.thr0, a.thr1, a.all0, a.all1, acc);
}

// Fields 4 j + p, j = J .. 5, of the four words, at bit 12 j: the masks' bits
// once they are moved up by 3 p.
template <int J, int ROUNDS>
__device__ __forceinline__ void ci_part(const CiCalls& calls, int p, const SweepArgs& a, ItemMasks& acc)
{
    if constexpr (4 * J < kFields) {
        if (4 * J + 3 < kFields || 4 * J + p < kFields) {
            uint32_t rnd[4];
            calls.template call<ROUNDS>(4 * J + p, a.rk, rnd);
#pragma unroll
            for (int e = 0; e < 4; ++e) accept_insert<(12 * J) & 31>(acc.m[e][12 * J / 32], rnd[e], a.thr0, a.thr1);
        }
        ci_part<J + 1, ROUNDS>(calls, p, a, acc);
    }
}

// The masks (lo, hi) of word row 4q + p, of which each of the block's four warps
// p draws the fields 4 j + p for all four rows (`parts`: [warp][row][lane]).
// Every thread of the block.
template <int ROUNDS>
__device__ __forceinline__ uint2 ci_masks_split(const uint4* tab, uint2 (*parts)[4][kCiBlockX], int p, int x, int m,
                                                uint64_t t, const SweepArgs& a)
{
    CiCalls calls;
    calls.keys = tab;
    mul_hilo(kPhiloxM0, philox_first_key((uint32_t)t, a.rk) ^ (uint32_t)m, calls.hi, calls.lo);
    ItemMasks acc;
#pragma unroll
    for (int e = 0; e < 4; ++e) acc.m[e][0] = acc.m[e][1] = 0;
    ci_part<0, ROUNDS>(calls, p, a, acc);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint64_t v = ((uint64_t)acc.m[e][1] << 32 | acc.m[e][0]) << (3 * p);
        parts[p][e][x] = make_uint2((uint32_t)v, (uint32_t)(v >> 32));
    }
    __syncthreads();
    uint64_t all = (((uint64_t)a.all1 << 32 | a.all1) & kAllFields) |
                   ((((uint64_t)a.all0 << 32 | a.all0) & kAllFields) << 1);
    uint2 r = make_uint2((uint32_t)all, (uint32_t)(all >> 32));
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        r.x |= parts[w][p][x].x;
        r.y |= parts[w][p][x].y;
    }
    return r;
}

// The update of one word (flip_half on both halves): s, its four neighbours
// and the masks (lo, hi) of the word.
__device__ __forceinline__ uint64_t ci_flip(uint64_t s, uint64_t xu, uint64_t xd, uint64_t xl, uint64_t xr,
                                            uint32_t mlo, uint32_t mhi)
{
    const uint32_t lo = flip_half((uint32_t)s, (uint32_t)xu, (uint32_t)xd, (uint32_t)xl, (uint32_t)xr, mlo,
                                  __funnelshift_r(mlo, mhi, 1), (uint32_t)kAllFields);
    const uint32_t hi = flip_half((uint32_t)(s >> 32), (uint32_t)(xu >> 32), (uint32_t)(xd >> 32),
                                  (uint32_t)(xl >> 32), (uint32_t)(xr >> 32), mhi, mhi >> 1,
                                  (uint32_t)(kAllFields >> 32));
    return (uint64_t)hi << 32 | lo;
}

// Anti-aligned bonds of the updated word and the up spins of it and `other`.
__device__ __forceinline__ void ci_count(uint64_t s, uint64_t xu, uint64_t xd, uint64_t xl, uint64_t xr,
                                         uint64_t other, uint32_t& anti, uint32_t& up)
{
    // three fields of one spin bit each fit one field
    anti += __popcll((s ^ xu) | (s ^ xd) << 1 | (s ^ xl) << 2) + __popcll(s ^ xr);
    up += __popcll(s | other << 1);
}

}  // namespace
}  // namespace ising
