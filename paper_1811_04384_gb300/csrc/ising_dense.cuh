// The dense form of a row-packed lattice inside the path kernels that keep it
// on chip (cluster and on-chip paths): one bit per spin, 32 sites of a
// colour-row per 32-bit word,
//   bit b of word w of colour-row (c, i) = up spin of site m = 32 w + b,
// with the bits past m = L/2 - 1 zero.  The 3-bit fields of the lattice's own
// words (Sec. 3) leave room for the neighbour sum of Eq. 3, which the bitwise
// form does not need: a dense word holds 32 sites per logic operation where
// half a packed word holds 10.5, takes a third of the shared memory, and the
// horizontal neighbour is one funnel shift.  The accept masks of a dense word
// are two words, r < thr1 and r < thr0.
#pragma once
#include <cstdint>

#include "ising_device.cuh"

namespace ising {

struct DenseGeom {
    int L;
    int W;        // words per colour-row = ceil((L/2) / 32)
    int P;        // row pitch in words: W rounded up to even (pad words stay zero)
    int lb;       // live bits of the last word (1..32)
};

inline DenseGeom dense_geom(int L)
{
    DenseGeom d;
    d.L = L;
    d.W = (L / 2 + 31) / 32;
    d.P = (d.W + 1) & ~1;
    d.lb = L / 2 - 32 * (d.W - 1);
    return d;
}

__device__ __forceinline__ uint32_t dense_live(const DenseGeom& d, int w)
{
    return w < d.W - 1 ? 0xffffffffu : (w == d.W - 1 ? 0xffffffffu >> (32 - d.lb) : 0u);
}

// Bits 3k, k = 0..20, of a packed word moved to bits k, and back.
__device__ __forceinline__ uint32_t pack_fields(uint64_t x)
{
    x &= kSpinBits;
    x = (x | x >> 2) & 0x10c30c30c30c30c3ull;
    x = (x | x >> 4) & 0x100f00f00f00f00full;
    x = (x | x >> 8) & 0x001f0000ff0000ffull;
    x = (x | x >> 16) & 0x001f00000000ffffull;
    x = (x | x >> 32) & 0x00000000001fffffull;
    return (uint32_t)x;
}

__device__ __forceinline__ uint64_t spread_fields(uint32_t v)
{
    uint64_t x = v & 0x1fffffu;
    x = (x | x << 32) & 0x001f00000000ffffull;
    x = (x | x << 16) & 0x001f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & kSpinBits;
    return x;
}

// Dense word w of a row of g.W packed words at index `row` of the array.
__device__ __forceinline__ uint32_t dense_from_packed(const uint64_t* words, uint64_t row, const Geom& g, int w)
{
    const uint64_t n = lattice_words(g);
    const int q = 32 * w / kFields, off = 32 * w - kFields * q;
    uint64_t v = 0;
    if (q < g.W) v = pack_fields(word_ld<false>(words, row + (uint64_t)q, n, __LINE__)) >> off;
    if (q + 1 < g.W)
        v |= (uint64_t)pack_fields(word_ld<false>(words, row + (uint64_t)q + 1, n, __LINE__)) << (kFields - off);
    if (q + 2 < g.W && 2 * kFields - off < 32)
        v |= (uint64_t)pack_fields(word_ld<false>(words, row + (uint64_t)q + 2, n, __LINE__)) << (2 * kFields - off);
    return (uint32_t)v;
}

// Packed word w from the dense words d0, d1 that hold its fields 21 w .. 21 w + 20
// (d0 at index 21 w / 32, d1 the next one or 0).
__device__ __forceinline__ uint64_t packed_from_dense(uint32_t d0, uint32_t d1, int w)
{
    return spread_fields(__funnelshift_r(d0, d1, (kFields * w) & 31));
}

// Anti-aligned bonds (four per updated word) and up spins (the word's and its
// same-column neighbour's) of dense words.  Bits are added by three-input adders
// (sum, carry) and counted as ones, twos and fours: a population count takes
// four times the issue slots of a logic operation.
struct DenseCount {
    uint32_t ones = 0, twos = 0, fours = 0, up1 = 0, up2 = 0;
    __device__ __forceinline__ void add(uint32_t s, uint32_t u, uint32_t d, uint32_t h0, uint32_t h1, uint32_t live)
    {
        constexpr int kSum = kLutA ^ kLutB ^ kLutC, kCarry = (kLutA & kLutB) | (kLutA & kLutC) | (kLutB & kLutC);
        const uint32_t a = s ^ u, b = s ^ d, c = s ^ h0, e = (s ^ h1) & live;
        const uint32_t t1 = lop3<kCarry>(ones, a, b), o = lop3<kSum>(ones, a, b), t2 = lop3<kCarry>(o, c, e);
        ones = lop3<kSum>(o, c, e);
        fours += __popc(lop3<kCarry>(twos, t1, t2));
        twos = lop3<kSum>(twos, t1, t2);
        up2 += __popc(lop3<kCarry>(up1, s, h0));
        up1 = lop3<kSum>(up1, s, h0);
    }
    __device__ __forceinline__ uint32_t anti() const { return __popc(ones) + 2 * __popc(twos) + 4 * fours; }
    __device__ __forceinline__ uint32_t up() const { return __popc(up1) + 2 * up2; }
};

// Draws of fields k .. N - 1 of the FirstTable column for the four rows of a
// row group, into bits k .. N - 1.
template <int k, int N, int ROUNDS, typename Calls>
struct DenseLoop {
    __device__ __forceinline__ static void run(const Calls& calls, const PhiloxKeys& rk, uint32_t (&m1)[4],
                                               uint32_t (&m0)[4], uint32_t thr0, uint32_t thr1)
    {
        if constexpr (k < N) {
            uint32_t rnd[4];
            calls.template call<ROUNDS>(k, rk, rnd);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                accept_bit<k>(m1[e], rnd[e], thr1);
                accept_bit<k>(m0[e], rnd[e], thr0);
            }
            DenseLoop<k + 1, N, ROUNDS, Calls>::run(calls, rk, m1, m0, thr0, thr1);
        }
    }
};

constexpr int kDenseStripWords = 8;      // most words of a strip of the dense mask draws

struct DenseFirst {
    const uint2* col;
    __device__ __forceinline__ void get(int k, uint32_t& hi, uint32_t& lo) const
    {
        const uint2 e = col[k * kDenseStripWords];
        hi = e.x;
        lo = e.y;
    }
};

// Where the masks of row 4 grp + e, word w of a half-sweep go, in words:
// masks[half * plane + grp * group + e * row + w].
struct DenseOut {
    uint32_t group, row, plane;
};

// The accept masks of sweeps t0 + 1 .., half-sweep by half-sweep (half =
// 2 sweep + colour), one 64-bit word per dense word: r < thr1 in the low half,
// r < thr0 in the high half, 0 on dead bits and pad words, set where the
// threshold is 2^32.  A block owns consecutive items (row group, word) of one
// strip, as in half_sweep_kernel.
// SPLIT = 1: a grid layer per sweep, a thread draws a whole word for both
// colours from one table of first products.  SPLIT = 4, for the on-chip warp's
// lattices of at most 64 items and the cluster path's short draws
// (kSplitThreads), where that would leave most SMs without a warp and the others
// with a chain of 64 draws: a layer per half-sweep, and a thread draws a quarter
// of a word (a byte of each mask).  The draws of 10 sweeps of L = 64 are a chain
// of 8 calls then instead of 64 (a call of 10 sweeps on chip 24.1 -> 20.4 us); 1024
// sweeps of L = 64 take 4.1 us.  Without a split: 1,744 sites/ns at L = 2016.
template <int ROUNDS, int SPLIT>
__global__ void __launch_bounds__(128, 8)
dense_mask_draw_kernel(DenseGeom d, Strips st, SweepArgs a, uint64_t t0, DenseOut to, uint64_t* __restrict__ masks)
{
    constexpr int N = 32 / SPLIT;
    __shared__ uint2 tab[32 * kDenseStripWords];
    pdl_launch();      // a launch that applies these masks may start and load its lattice
    const uint32_t w0 = blockIdx.y * st.width;
    const bool last = blockIdx.y == st.n - 1u;
    const uint32_t width = last ? st.last : st.width, magic = last ? st.magic_last : st.magic;
    const uint32_t sweep = SPLIT == 1 ? blockIdx.z : blockIdx.z >> 1;
    const uint64_t t = t0 + sweep + 1;
    first_products<32, kDenseStripWords>(tab, w0, width, magic, philox_first_key((uint32_t)t, a.rk));
    const uint32_t thread = blockIdx.x * blockDim.x + threadIdx.x, q = thread / SPLIT, part = thread % SPLIT;
    const uint32_t grp = strip_group(q, magic), x = q - grp * width;
    const int w = (int)(w0 + x);
    if (grp * 4u >= (uint32_t)d.L) return;
    const uint32_t live = dense_live(d, w) >> (N * part);
    const int c0 = SPLIT == 1 ? 0 : blockIdx.z & 1;
    uint64_t out = (uint64_t)(2 * sweep + c0) * to.plane + grp * to.group + w;
#ifdef ISING_CHECKED
    const uint64_t n = (uint64_t)gridDim.z * (SPLIT == 1 ? 2 : 1) * to.plane;
#endif
#pragma unroll 1
    for (int c = c0; c < (SPLIT == 1 ? 2 : c0 + 1); ++c, out += to.plane) {
        uint32_t m1[4] = {0, 0, 0, 0}, m0[4] = {0, 0, 0, 0};
        if (live) {
            const RowCalls<DenseFirst> calls = {{tab + x + N * kDenseStripWords * part},
                                                philox_row_key(grp, (uint32_t)t, counter_high(t, c), a.rk)};
            DenseLoop<0, N, ROUNDS, RowCalls<DenseFirst>>::run(calls, a.rk, m1, m0, a.thr0, a.thr1);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (grp * 4u + e >= (uint32_t)d.L) continue;
            m1[e] = (m1[e] | a.all1) & live;
            m0[e] = (m0[e] | a.all0) & live;
            uint64_t* const word = masks + out + (uint64_t)e * to.row;
#ifdef ISING_CHECKED
            if (!check_index(out + (uint64_t)e * to.row, n, __LINE__)) continue;
#endif
            if constexpr (SPLIT == 1) {
                *word = (uint64_t)m0[e] << 32 | m1[e];
            } else {
                static_assert(N == 8, "a part is a byte");
                uint8_t* byte = reinterpret_cast<uint8_t*>(word) + part;
                byte[0] = (uint8_t)m1[e];
                byte[4] = (uint8_t)m0[e];
            }
        }
    }
}

}  // namespace ising
