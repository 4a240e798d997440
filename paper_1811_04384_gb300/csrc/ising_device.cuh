// Device code of the multi-spin Ising Metropolis path (sm_103a).
//
// Layout (multi-spin coding of Sec. 3, 3-bit fields, 000 = down, 001 = up, 21
// spins per 64-bit word, bit 63 zero).  The paper interleaves 21 rows of one
// column into a word and needs L = 21N; here the spins of one colour in one
// row are packed along the row, so any even L works:
//   colour c = (i + j) & 1, m = j >> 1 in [0, L/2) indexes the colour-c sites
//   of row i; word w of colour-row (c, i) holds m = 21 w + k in field k
//   (bits 3k .. 3k+2); the last word of a row holds `rlast` live fields and
//   its dead fields stay zero.  Array c is row-major, `P` words per row.
//
// Neighbours of a colour-c site (i, m): up/down are field m of the
// other-colour rows i-1 / i+1; left/right are fields m and m-1 of row i when
// (i + c) is even, fields m and m+1 when it is odd (periodic in m over L/2).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include "philox.cuh"

namespace ising {

constexpr int kFields = 21;
constexpr uint64_t kSpinBits = 0x1249249249249249ull;   // bit 3k, k = 0..20
constexpr int kCountSlots = 32;                          // spread of the E/M atomics

struct Geom {
    int L;          // lattice side (even, >= 4)
    int W;          // words per colour-row = ceil((L/2) / 21)
    int P;          // row pitch in words (W rounded up to even)
    int rlast;      // live fields in the last word of a row (1..21)
};

// Per-launch constants of one half-sweep.
struct SweepArgs {
    const uint64_t* t_base;    // device: sweep counter before this chunk, or null ...
    uint64_t t0;               // ... and then the same on the host
    uint32_t t_off;            // this half-sweep belongs to sweep (t_base ? *t_base : t0) + t_off
    uint32_t thr0, thr1;       // integer thresholds clamped to 2^32 - 1 ...
    uint32_t all0, all1;       // ... and ~0u where the threshold is 2^32
    uint32_t rounds;           // Philox rounds of the sweep draws: 10 (default) or 7 (opt-in)
    PhiloxKeys rk;             // round keys of the key (lo32(seed), hi32(seed))
    unsigned long long* counts;  // E/M count slots of this record (RECORD only)
    const uint32_t* rec_base;    // device record index added to `counts` (graph replays), or null
};

// The 32 count slots a RECORD launch adds to: `counts`, moved on by
// *rec_base records when a replayed graph picks its slot on the device.
__device__ __forceinline__ unsigned long long* record_counts(const SweepArgs& a)
{
    return a.rec_base ? a.counts + (size_t)(*a.rec_base) * 2 * kCountSlots : a.counts;
}

// Programmatic dependent launch: a half-sweep launched with programmatic
// stream serialization lets the next half-sweep be launched and its blocks be
// placed as soon as every block of this one has started (launch_dependents),
// and waits, before its first read of device memory, until the previous grid
// has completed and its writes are visible (wait).  Both are no-ops in a
// plain launch.  What a block does before the wait (its draws, which need
// launch operands only) overlaps the end of the previous grid.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The sweep number of a half-sweep, read before the wait: the device counter
// is advanced only by a plain launch at the end of a chunk (or graph), which
// the half-sweeps of the next chunk start after.
__device__ __forceinline__ uint64_t sweep_number(const SweepArgs& a) { return (a.t_base ? *a.t_base : a.t0) + a.t_off; }

// ---- Checked build (compiled with -DISING_CHECKED) -------------------------
// Every lattice-word access of the sweep routines goes through word_ld /
// word_st with the length of the array it indexes.  In a checked build an
// index at or past that length is not accessed (a load gives 0, a store is
// dropped) and the first such index is recorded, with the source line of the
// access, in this translation unit's device word g_check_word; the host reads
// and clears the words of every translation unit (ising_check_status).
// Nothing traps or asserts, so a bad index leaves the context usable.  In the
// normal build these are plain accesses.
#ifdef ISING_CHECKED
static __device__ unsigned long long g_check_word;

__device__ __forceinline__ bool check_index(uint64_t idx, uint64_t n, uint32_t line)
{
    if (idx < n) return true;
    atomicCAS(&g_check_word, 0ull, (1ull << 63) | ((uint64_t)(line & 0x7FFFFFu) << 40) | (idx & 0xFFFFFFFFFFull));
    return false;
}

// Host side: this translation unit's word, read and cleared (registered with
// the library's list of readers when the library loads).
bool register_check_reader(int (*reader)(unsigned long long*));
static int read_check_word(unsigned long long* out)
{
    const unsigned long long zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(out, g_check_word, sizeof(zero));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_check_word, &zero, sizeof(zero));
    return e == cudaSuccess ? 0 : -1;
}
static const bool g_check_reader_registered = register_check_reader(&read_check_word);
#endif

// A lattice word p[idx] of an array of n words: through the read-only cache
// (LDG) or a plain load.
template <bool LDG>
__device__ __forceinline__ uint64_t word_ld(const uint64_t* p, uint64_t idx, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(idx, n, line)) return 0;
#endif
    return LDG ? __ldg(p + idx) : p[idx];
}

__device__ __forceinline__ void word_st(uint64_t* p, uint64_t idx, uint64_t v, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(idx, n, line)) return;
#endif
    p[idx] = v;
}

__device__ __forceinline__ uint32_t half_ld(const uint32_t* p, uint64_t idx, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(idx, n, line)) return 0;
#endif
    return p[idx];
}

__device__ __forceinline__ void half_st(uint32_t* p, uint64_t idx, uint32_t v, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(idx, n, line)) return;
#endif
    p[idx] = v;
}

// Four 32-bit words from p[idx] on, idx a multiple of four.
__device__ __forceinline__ uint4 vector_ld(const uint32_t* p, uint32_t idx, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index((uint64_t)idx + 3, n, line)) return make_uint4(0, 0, 0, 0);
#endif
    return *reinterpret_cast<const uint4*>(p + idx);
}

// The word, or the 32-bit half of one, at byte offset `o` of an array of n words.
__device__ __forceinline__ uint64_t byte_ld64(const uint64_t* p, uint32_t o, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(o / 8u, n, line)) return 0;
#endif
    return *reinterpret_cast<const uint64_t*>(reinterpret_cast<const char*>(p) + o);
}

__device__ __forceinline__ uint32_t byte_ld32(const uint64_t* p, uint32_t o, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(o / 4u, 2 * n, line)) return 0;
#endif
    return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(p) + o);
}

__device__ __forceinline__ void byte_st64(uint64_t* p, uint32_t o, uint64_t v, uint64_t n, uint32_t line)
{
#ifdef ISING_CHECKED
    if (!check_index(o / 8u, n, line)) return;
#endif
    *reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(p) + o) = v;
}

__device__ __forceinline__ uint64_t lattice_words(const Geom& g) { return (uint64_t)g.L * (uint64_t)g.P; }

__device__ __forceinline__ int wrap_row(int i, int L)
{
    return i < 0 ? i + L : (i >= L ? i - L : i);
}

__device__ __forceinline__ uint64_t live_mask(const Geom& g, int w)
{
    return (w == g.W - 1) ? (kSpinBits & ((g.rlast == kFields) ? ~0ull : ((1ull << (3 * g.rlast)) - 1ull)))
                          : kSpinBits;
}

// Block-wide sum of two counters, added with one atomic each to target[0..1].
__device__ __forceinline__ void block_add_counts(unsigned long long* target, uint32_t anti, uint32_t up)
{
    __shared__ unsigned int s_anti[32], s_up[32];
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    const int nthreads = blockDim.x * blockDim.y;
    const int lane = tid & 31, warp = tid >> 5;
    anti = __reduce_add_sync(0xffffffffu, anti);
    up = __reduce_add_sync(0xffffffffu, up);
    if (lane == 0) { s_anti[warp] = anti; s_up[warp] = up; }
    __syncthreads();
    if (warp == 0) {
        const int nw = (nthreads + 31) >> 5;
        unsigned int a = (lane < nw) ? s_anti[lane] : 0u;
        unsigned int u = (lane < nw) ? s_up[lane] : 0u;
        a = __reduce_add_sync(0xffffffffu, a);
        u = __reduce_add_sync(0xffffffffu, u);
        if (lane == 0) {
            atomicAdd(target + 0, (unsigned long long)a);
            atomicAdd(target + 1, (unsigned long long)u);
        }
    }
}

// d = LUT(a, b, c) bit by bit, LUT over kLutA, kLutB, kLutC: one instruction.
constexpr int kLutA = 0xF0, kLutB = 0xCC, kLutC = 0xAA;
template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT & 0xFF));
    return d;
}

// The Metropolis step of Sec. 2 on one 32-bit half of a word: s the own
// spins, u, d, h0, h1 the four neighbours', p the sites with r < thr1, q
// those with r < thr0, live the spin bits.  With x_n = s ^ n (anti-aligned),
// A = x_u | x_d, B = x_u & x_d, C = x_h0 | x_h1, D = x_h0 & x_h1 (Eq. 3
// summed bitwise), two or more anti-aligned neighbours (dE <= 0, Table 1) are
// B | D | A & C and one or more A | C.  thr0 <= thr1, so q implies p, and
//   accept = B | D | A & C | (A | C) & p | q = (B | D | q) | majority(A, C, p):
// eight three-input operations.
__device__ __forceinline__ uint32_t flip_half(uint32_t s, uint32_t u, uint32_t d, uint32_t h0, uint32_t h1,
                                              uint32_t p, uint32_t q, uint32_t live)
{
    constexpr int kOr = (kLutA ^ kLutB) | (kLutA ^ kLutC), kAnd = (kLutA ^ kLutB) & (kLutA ^ kLutC);
    const uint32_t A = lop3<kOr>(s, u, d), B = lop3<kAnd>(s, u, d);
    const uint32_t C = lop3<kOr>(s, h0, h1), D = lop3<kAnd>(s, h0, h1);
    const uint32_t e = lop3<(kLutA | kLutB | kLutC)>(B, D, q);
    const uint32_t m = lop3<(kLutA & kLutB) | (kLutA & kLutC) | (kLutB & kLutC)>(A, C, p);
    return s ^ lop3<(kLutA | kLutB) & kLutC>(e, m, live);
}

// flip_half where p and q are zero off the live bits and h1 alone of the
// neighbours can be set there: A, B and D are zero there, so nothing flips.
__device__ __forceinline__ uint32_t flip_all(uint32_t s, uint32_t u, uint32_t d, uint32_t h0, uint32_t h1, uint32_t p,
                                             uint32_t q)
{
    constexpr int kOr = (kLutA ^ kLutB) | (kLutA ^ kLutC), kAnd = (kLutA ^ kLutB) & (kLutA ^ kLutC);
    const uint32_t A = lop3<kOr>(s, u, d), B = lop3<kAnd>(s, u, d);
    const uint32_t C = lop3<kOr>(s, h0, h1), D = lop3<kAnd>(s, h0, h1);
    const uint32_t e = lop3<(kLutA | kLutB | kLutC)>(B, D, q);
    const uint32_t m = lop3<(kLutA & kLutB) | (kLutA & kLutC) | (kLutB & kLutC)>(A, C, p);
    return lop3<(kLutA ^ (kLutB | kLutC))>(s, e, m);
}

// Anti-aligned bonds of the updated half word s with its four neighbours, and
// its up spins plus those of h0, added to anti / up.  Two spin-bit words share
// one population count (x + 2 y: the fields are three bits wide).
__device__ __forceinline__ void count_half(uint32_t s, uint32_t u, uint32_t d, uint32_t h0, uint32_t h1,
                                           uint32_t live, uint32_t& anti, uint32_t& up)
{
    const uint32_t xh1 = lop3<(kLutA ^ kLutB) & kLutC>(s, h1, live);
    anti += __popc((s ^ u) + 2u * (s ^ d)) + __popc((s ^ h0) + 2u * xh1);
    up += __popc(s + 2u * h0);
}

// Accept masks of an item (4 rows x 1 word of one colour): per row and 32-bit
// half, r < thr1 of field k at bit 3k of the word and r < thr0 at bit 3k + 1.
// One accumulator holds both (their other bits fall on no spin bit), so a row
// needs two registers.
struct ItemMasks {
    uint32_t m[4][2];   // [row][half]
};

// The inserts are predicated PTX, so a compare result never becomes a 0/1
// value and the bit is an immediate.  On GB300 the Philox products and the
// ALU share issue: a product takes four cycles of the multiply pipe and two
// of the ALU's, any ALU operation two.  The products, XORs and compares
// already fill those, so the inserts have to go to the multiply pipe: as an
// OR into bits that are known to be zero they do (the compiler turns it into
// an add there; as an XOR they stayed on the ALU, 1,243 against 1,394
// spin-updates/ns at L = 16384).
template <int B>
__device__ __forceinline__ void accept_bit(uint32_t& acc, uint32_t r, uint32_t thr)
{
    asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}"
        : "+r"(acc) : "r"(r), "r"(thr), "n"(1u << B));
}

template <int B>
__device__ __forceinline__ void accept_insert(uint32_t& acc, uint32_t r, uint32_t thr0, uint32_t thr1)
{
    accept_bit<B>(acc, r, thr1);
    accept_bit<B + 1>(acc, r, thr0);
}

// The first Philox products of an item's fields: computed (m = m0 + k), or
// read from a block's shared table (first_products).
struct FirstDirect {
    uint32_t key, m0;
    __device__ __forceinline__ void get(int k, uint32_t& hi, uint32_t& lo) const
    {
        mul_hilo(kPhiloxM0, key ^ (m0 + (uint32_t)k), hi, lo);
    }
};
constexpr int kStripWords = 16;   // most words of a strip
struct FirstTable {
    const uint2* col;             // the item's word in the table
    __device__ __forceinline__ void get(int k, uint32_t& hi, uint32_t& lo) const
    {
        const uint2 e = col[k * kStripWords];
        hi = e.x;
        lo = e.y;
    }
};

// The calls of an item's 21 fields, one row group: from the row group's key and
// the fields' first products.
template <typename First>
struct RowCalls {
    First first;
    PhiloxRowKey pk;
    template <int ROUNDS>
    __device__ __forceinline__ void call(int k, const PhiloxKeys& rk, uint32_t rnd[4]) const
    {
        uint32_t hi, lo;
        first.get(k, hi, lo);
        philox_row_tail<ROUNDS>(pk, rk, hi, lo, rnd);
    }
};

// Fields k .. 20 (compile-time k: immediate bit masks); call k gives the draws
// of field k of four rows.
template <int k, int ROUNDS, typename Calls>
struct FieldLoop {
    __device__ __forceinline__ static void run(const Calls& calls, const PhiloxKeys& rk, ItemMasks& acc,
                                               uint32_t thr0, uint32_t thr1)
    {
        uint32_t rnd[4];
        calls.template call<ROUNDS>(k, rk, rnd);
        constexpr int half = k <= 10 ? 0 : 1;
        constexpr int B = k <= 10 ? 3 * k : 3 * k - 32;
#pragma unroll
        for (int e = 0; e < 4; ++e) accept_insert<B>(acc.m[e][half], rnd[e], thr0, thr1);
        FieldLoop<k + 1, ROUNDS, Calls>::run(calls, rk, acc, thr0, thr1);
    }
};
template <int ROUNDS, typename Calls>
struct FieldLoop<kFields, ROUNDS, Calls> {
    __device__ __forceinline__ static void run(const Calls&, const PhiloxKeys&, ItemMasks&, uint32_t, uint32_t) {}
};

// The masks of the 21 fields of `calls` (Sec. 2 steps 2-3).
template <int ROUNDS, typename Calls>
__device__ __forceinline__ void draw_fields(const Calls& calls, const PhiloxKeys& rk, uint32_t thr0, uint32_t thr1,
                                            uint32_t all0w, uint32_t all1w, ItemMasks& acc)
{
#pragma unroll
    for (int e = 0; e < 4; ++e) acc.m[e][0] = acc.m[e][1] = 0;
    FieldLoop<0, ROUNDS, Calls>::run(calls, rk, acc, thr0, thr1);
    if (all1w | all0w) {     // a threshold of 2^32 accepts always
        const uint64_t a = ((((uint64_t)all1w << 32 | all1w) & kSpinBits)) |
                           ((((uint64_t)all0w << 32 | all0w) & kSpinBits) << 1);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            acc.m[e][0] |= (uint32_t)a;
            acc.m[e][1] |= (uint32_t)(a >> 32);
        }
    }
}

// The high counter word of colour c at sweep t.
__device__ __forceinline__ uint32_t counter_high(uint64_t t, int c) { return ((uint32_t)(t >> 32) << 1) | (uint32_t)c; }

// The masks of row group grp at sweep t, colour `colour` (one Philox call
// covers the four rows of one field).
template <int ROUNDS, typename First>
__device__ __forceinline__ void draw_item(const First& first, uint32_t grp, uint64_t t, int colour,
                                          const PhiloxKeys& rk, uint32_t thr0, uint32_t thr1, uint32_t all0w,
                                          uint32_t all1w, ItemMasks& acc)
{
    const RowCalls<First> calls = {first, philox_row_key(grp, (uint32_t)t, counter_high(t, colour), rk)};
    draw_fields<ROUNDS>(calls, rk, thr0, thr1, all0w, all1w, acc);
}

// Update (and/or record) rows 4 grp .. 4 grp + 3 (those below L) of word
// column w of colour C with the masks `acc` (same-colour sites are never
// neighbours).  Byte offsets are 32-bit (a colour array has less than 2^28
// bytes).  Only rows 0 and 1 of a group can exist alone (L even): the
// missing rows then read rows 0 and 1 of the lattice and are not stored.
// The side word gives one field only, so only its half is read: field 20
// (or the row's last field across the wrap) of the word to the left, shifted
// down to field 0, or field 0 of the word to the right, moved up by a
// multiply.  UPDATE = false skips the flip (measurement only).  RECORD adds
// the anti-aligned bond count of the (updated) colour-1 words and the up-spin
// count of both colours to anti / up: E = 2 anti - 2 L^2, M = 2 up - L^2.
template <int C, bool UPDATE, bool RECORD>
__device__ __forceinline__ void apply_item(uint64_t* own, const uint64_t* other, const Geom& g, uint32_t grp,
                                           uint32_t w, const ItemMasks& acc, uint32_t& anti, uint32_t& up)
{
    const uint32_t P8 = (uint32_t)g.P * 8u, LP8 = (uint32_t)g.L * P8, row0 = grp * 4u, w8 = w * 8u;
    const bool two = row0 + 2u >= (uint32_t)g.L;                       // rows 0 and 1 only
    // byte offsets of rows row0 - 1 .. row0 + 4 (periodic), word w
    const uint32_t o1 = row0 * P8 + w8, o2 = o1 + P8, o3 = o2 + P8 - (two ? LP8 : 0u), o4 = o3 + P8;
    const uint32_t o0 = o1 - P8 + (row0 == 0u ? LP8 : 0u);
    const uint32_t o5 = o4 + P8 - (row0 + 4u == (uint32_t)g.L ? LP8 : 0u);
    const bool first = w == 0u, last = w == (uint32_t)g.W - 1u;
    const uint32_t lastbit = 3u * (uint32_t)(g.rlast - 1);             // the row's last live field
    const uint32_t left = first ? (uint32_t)(g.W - 1) * 8u + (lastbit >= 32u ? 4u : 0u) : (uint32_t)-4;
    const uint32_t lsh = first ? (lastbit & 31u) : 28u;
    const uint32_t right = last ? 0u - w8 : 8u;
    const uint32_t mul_lo = last && lastbit < 32u ? 1u << lastbit : 0u;
    const uint32_t mul_hi = last ? (lastbit >= 32u ? 1u << (lastbit & 31u) : 0u) : 1u << 28;
    const uint64_t n = lattice_words(g);
    uint64_t oc[6], sw[4];
    uint32_t side[4];
    oc[0] = byte_ld64(other, o0, n, __LINE__);
    oc[1] = byte_ld64(other, o1, n, __LINE__);
    oc[2] = byte_ld64(other, o2, n, __LINE__);
    oc[3] = byte_ld64(other, o3, n, __LINE__);
    oc[4] = byte_ld64(other, o4, n, __LINE__);
    oc[5] = byte_ld64(other, o5, n, __LINE__);
    const uint32_t even = C == 0 ? left : right, odd = C == 0 ? right : left;
    side[0] = byte_ld32(other, o1 + even, n, __LINE__);
    side[1] = byte_ld32(other, o2 + odd, n, __LINE__);
    side[2] = byte_ld32(other, o3 + even, n, __LINE__);
    side[3] = byte_ld32(other, o4 + odd, n, __LINE__);
    sw[0] = byte_ld64(own, o1, n, __LINE__);
    sw[1] = byte_ld64(own, o2, n, __LINE__);
    sw[2] = byte_ld64(own, o3, n, __LINE__);
    sw[3] = byte_ld64(own, o4, n, __LINE__);
    const uint64_t live64 = live_mask(g, (int)w);
    const uint32_t live[2] = {(uint32_t)live64, (uint32_t)(live64 >> 32)};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t s[2] = {(uint32_t)sw[r], (uint32_t)(sw[r] >> 32)};
        const uint32_t u[2] = {(uint32_t)oc[r], (uint32_t)(oc[r] >> 32)};
        const uint32_t h0[2] = {(uint32_t)oc[r + 1], (uint32_t)(oc[r + 1] >> 32)};
        const uint32_t d[2] = {(uint32_t)oc[r + 2], (uint32_t)(oc[r + 2] >> 32)};
        // the horizontal neighbour at m - 1 (row + C even: row0 is a multiple of 4) or m + 1: the other
        // colour's word moved by one field (bit 63 and dead fields are masked by live)
        uint32_t h1[2], sn[2] = {s[0], s[1]};
        if (((r + C) & 1) == 0) {
            h1[0] = h0[0] * 8u + (side[r] >> lsh);
            h1[1] = __funnelshift_l(h0[0], h0[1], 3);
        } else {
            h1[0] = __funnelshift_r(h0[0], h0[1], 3) + side[r] * mul_lo;
            h1[1] = (h0[1] >> 3) + side[r] * mul_hi;
        }
        if (UPDATE) {
            sn[0] = flip_half(s[0], u[0], d[0], h0[0], h1[0], acc.m[r][0],
                              __funnelshift_r(acc.m[r][0], acc.m[r][1], 1), live[0]);
            sn[1] = flip_half(s[1], u[1], d[1], h0[1], h1[1], acc.m[r][1], acc.m[r][1] >> 1, live[1]);
        }
        if (r < 2 || !two) {
            if (UPDATE) {
                const uint32_t o = r == 0 ? o1 : (r == 1 ? o2 : (r == 2 ? o3 : o4));
                byte_st64(own, o, (uint64_t)sn[1] << 32 | sn[0], n, __LINE__);
            }
            if (RECORD) {
                count_half(sn[0], u[0], d[0], h0[0], h1[0], live[0], anti, up);
                count_half(sn[1], u[1], d[1], h0[1], h1[1], live[1], anti, up);
            }
        }
    }
}

// ---- Strips: the items of a launch --------------------------------------
// The thread items (group of 4 rows x word) are numbered strip by strip: a
// strip is up to kStripWords consecutive word columns of all row groups, and
// item q of a strip of `width` words is word q % width of group q / width.  A
// block owns consecutive items of one strip, so its row groups share their
// words' columns m = 21 w + k and with them the first Philox product of each
// (first_products): 15 products per call instead of 16, and no index XOR.
// Measured on GB300 at L = 16384 (one colour, launches back to back): 1,487
// spin-updates/ns against 1,335-1,370 with the items in row order and each
// call's own first product (26.1 against 28.1 cycles per site and scheduler,
// with the word logic and index arithmetic trimmed at the same time).  Strips
// of at most 32 / 24 / 20 / 16 / 12 words (blocks of 128, sweeps without
// records): 1,537 / 1,551 / 1,558 / 1,567 / 1,574, but L = 2016: 1,136 /
// 1,144 / 1,153 / 1,159 / 1,124; 16 words are 128 bytes of a row.
struct Strips {
    uint32_t n;              // strips
    uint32_t width, last;    // words of a strip, of the last one
    uint32_t magic, magic_last;   // q / width = hi32(q * magic); 0: width 1
};

__device__ __forceinline__ uint32_t strip_group(uint32_t q, uint32_t magic) { return magic ? __umulhi(q, magic) : q; }

// All threads of the block: the first products of fields 0 .. FIELDS - 1 of
// words w0 .. w0 + width - 1 at a sweep (key: philox_first_key), field k of
// word w0 + x in tab[k * STRIDE + x].  The threads fill whole columns of a
// field at a time (blockDim / width fields per pass).
template <int FIELDS, int STRIDE>
__device__ __forceinline__ void first_products(uint2* tab, uint32_t w0, uint32_t width, uint32_t magic, uint32_t key)
{
    const uint32_t k0 = strip_group(threadIdx.x, magic), x = threadIdx.x - k0 * width;
    const uint32_t step = strip_group(blockDim.x, magic);      // >= 2: blocks have at least 32 threads
    uint32_t m = (w0 + x) * (uint32_t)FIELDS + k0;
    if (k0 < step)
        for (uint32_t k = k0; k < (uint32_t)FIELDS; k += step, m += step) {
            uint32_t hi, lo;
            mul_hilo(kPhiloxM0, key ^ m, hi, lo);
            tab[k * STRIDE + x] = make_uint2(hi, lo);
        }
    __syncthreads();
}

// Draw and update in one step without a table (the on-chip kernel that draws
// its own masks).
template <int C, bool RECORD, int ROUNDS>
__device__ __forceinline__ void sweep_item(uint64_t* own, const uint64_t* other, const Geom& g, uint32_t grp,
                                           uint32_t w, uint64_t t, const SweepArgs& a, uint32_t& anti, uint32_t& up)
{
    ItemMasks acc;
    const FirstDirect first = {philox_first_key((uint32_t)t, a.rk), w * (uint32_t)kFields};
    draw_item<ROUNDS>(first, grp, t, C, a.rk, a.thr0, a.thr1, a.all0, a.all1, acc);
    apply_item<C, true, RECORD>(own, other, g, grp, w, acc, anti, up);
}

// ---- Split forms of an item's step ---------------------------------------
// The work of an item in two parts: its accept masks (the Philox draws
// against the thresholds; they depend on the site, sweep and colour only,
// never on the spins) and their application to the item's rows.  So the
// masks can be drawn by other threads than the ones that apply them, or
// before the spins they apply to exist: F lanes per item on the launch path
// for lattices too small to fill the GPU with one thread per item, and all
// masks of a run drawn beforehand for the on-chip path.  The draws and the
// accept rule are those of draw_item and apply_item, so the results are
// bit-identical.  All
// lanes of a warp must call the lane forms (shuffles); an item past the end
// (`valid` = false) is drawn as item 0 and never applied.

// F lanes per item (F = 2, 4 or 8; aligned groups of the warp): lane q draws
// the fields k = q + jF, collects its accept bits at bit 3jF (compile-time
// positions), shifts them by 3q to bit 3k and OR-merges the F lanes' masks
// with shuffles.  Every lane of the group gets all masks.
template <int F, int ROUNDS = 10>
__device__ __forceinline__ void item_masks_lanes(const Geom& g, int item, int q, uint64_t t, int colour,
                                                 const PhiloxKeys& rk, uint32_t thr0, uint32_t thr1,
                                                 uint64_t a1[4], uint64_t a0[4])
{
    static_assert(F == 2 || F == 4 || F == 8, "F: 2, 4 or 8 lanes per item");
    constexpr int J = (kFields + F - 1) / F;
    const int grp = item / g.W;
    const int w = item - grp * g.W;
    const uint32_t tl = (uint32_t)t;
    const uint32_t th = ((uint32_t)(t >> 32) << 1) | (uint32_t)colour;
    const PhiloxRowKey pk = philox_row_key((uint32_t)grp, tl, th, rk);
#pragma unroll
    for (int e = 0; e < 4; ++e) a1[e] = a0[e] = 0;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int k = q + j * F;
        if (k < kFields) {
            uint32_t r[4];
            philox_row<ROUNDS>(pk, rk, (uint32_t)(w * kFields + k), r);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (r[e] < thr1) a1[e] |= 1ull << (3 * j * F);
                if (r[e] < thr0) a0[e] |= 1ull << (3 * j * F);
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        a1[e] <<= 3 * q;
        a0[e] <<= 3 * q;
    }
#pragma unroll
    for (int d = 1; d < F; d <<= 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            a1[e] |= __shfl_xor_sync(0xffffffffu, a1[e], d);
            a0[e] |= __shfl_xor_sync(0xffffffffu, a0[e], d);
        }
    }
}

// Apply the masks m1 (r < thr1) and m0 (r < thr0) of row i, word w of colour
// C: the spin logic of apply_item for one row.  all0 / all1 are the "always"
// masks (thresholds of 2^32) and live the row's live spin bits.  RECORD adds
// the row's anti-aligned bonds and up spins to anti / up (colour 1).
template <int C, bool RECORD>
__device__ __forceinline__ void row_apply(uint64_t* __restrict__ own, const uint64_t* __restrict__ other,
                                          const Geom& g, int i, int w, uint64_t live, uint64_t m1, uint64_t m0,
                                          uint64_t all0, uint64_t all1, uint32_t& anti, uint32_t& up)
{
    const uint32_t P = (uint32_t)g.P;
    const uint32_t o = (uint32_t)i * P;
    const uint64_t n = lattice_words(g);
    const uint64_t s = word_ld<false>(own, o + (uint32_t)w, n, __LINE__);
    const uint64_t u = word_ld<false>(other, (uint32_t)wrap_row(i - 1, g.L) * P + (uint32_t)w, n, __LINE__);
    const uint64_t d = word_ld<false>(other, (uint32_t)wrap_row(i + 1, g.L) * P + (uint32_t)w, n, __LINE__);
    const uint64_t h0 = word_ld<false>(other, o + (uint32_t)w, n, __LINE__);
    // horizontal neighbour at m - 1 ((i + C) even) or m + 1 (odd), as in apply_item
    const bool left = ((i + C) & 1) == 0;
    const int ws = left ? ((w > 0) ? w - 1 : g.W - 1) : ((w < g.W - 1) ? w + 1 : 0);
    const int sh = (left ? (w > 0) : (w < g.W - 1)) ? 60 : 3 * (g.rlast - 1);
    const uint64_t side = word_ld<false>(other, o + (uint32_t)ws, n, __LINE__);
    const uint64_t h1 = left ? ((h0 << 3) | (side >> sh)) : ((h0 >> 3) | (side << sh));
    const uint64_t x1 = s ^ u, x2 = s ^ d, x3 = s ^ h0, x4 = s ^ h1;
    const uint64_t any = x1 | x2 | x3 | x4;
    const uint64_t ge2 = (x1 & x2) | (x3 & x4) | ((x1 ^ x2) & (x3 ^ x4));
    const uint64_t accept = ge2 | (any & (m1 | all1)) | (~any & (m0 | all0));
    const uint64_t s_new = s ^ (accept & live);
    word_st(own, o + (uint32_t)w, s_new, n, __LINE__);
    if (RECORD) {
        anti += __popcll((s_new ^ u) & live) + __popcll((s_new ^ d) & live)
              + __popcll((s_new ^ h0) & live) + __popcll((s_new ^ h1) & live);
        up += __popcll(s_new & live) + __popcll(h0 & live);
    }
}

// Apply the masks of an item of colour C: lane q of its group of F lanes
// updates rows q, q + F, ... below 4 (one code path for all lanes, the row's
// masks picked by selection).  RECORD adds the item's
// anti-aligned bonds and up spins to anti / up (colour 1).
template <int C, bool RECORD, int F>
__device__ __forceinline__ void item_apply(uint64_t* __restrict__ own, const uint64_t* __restrict__ other,
                                           const Geom& g, int item, bool valid, int q, const uint64_t a1[4],
                                           const uint64_t a0[4], uint32_t all0w, uint32_t all1w, uint32_t& anti,
                                           uint32_t& up)
{
    constexpr int STEP = F < 4 ? F : 4;
    if (!valid) return;
    const int grp = item / g.W;
    const int w = item - grp * g.W;
    const int row0 = grp * 4;
    const uint64_t live = live_mask(g, w);
    const uint64_t all0 = ((uint64_t)all0w << 32 | all0w) & live;
    const uint64_t all1 = ((uint64_t)all1w << 32 | all1w) & live;
#pragma unroll
    for (int e0 = 0; e0 < 4; e0 += STEP) {
        const int e = e0 + q;
        if (e >= 4 || e >= g.L - row0) break;
        const uint64_t m1 = e == 0 ? a1[0] : (e == 1 ? a1[1] : (e == 2 ? a1[2] : a1[3]));
        const uint64_t m0 = e == 0 ? a0[0] : (e == 1 ? a0[1] : (e == 2 ? a0[2] : a0[3]));
        row_apply<C, RECORD>(own, other, g, row0 + e, w, live, m1, m0, all0, all1, anti, up);
    }
}

// All accept masks of one item drawn by one thread, packed one word per row:
// packed[e] has r < thr1 of field k at bit 3k and r < thr0 at bit 3k + 1, each
// set where its threshold is 2^32.  For row_apply, m1 = packed and m0 =
// packed >> 1: their other bits fall on no spin bit.
template <int ROUNDS = 10>
__device__ __forceinline__ void item_masks_thread(const Geom& g, int item, uint64_t t, int colour, const SweepArgs& a,
                                                  uint64_t packed[4])
{
    const int grp = item / g.W;
    const int w = item - grp * g.W;
    ItemMasks acc;
    const FirstDirect first = {philox_first_key((uint32_t)t, a.rk), (uint32_t)w * kFields};
    draw_item<ROUNDS>(first, (uint32_t)grp, t, colour, a.rk, a.thr0, a.thr1, a.all0, a.all1, acc);
#pragma unroll
    for (int e = 0; e < 4; ++e) packed[e] = (uint64_t)acc.m[e][1] << 32 | acc.m[e][0];
}

// Masks of an item with F lanes; an item past the end is drawn as item 0.
template <int F, int ROUNDS = 10>
__device__ __forceinline__ void item_masks(const Geom& g, int item, bool valid, int q, uint64_t t, int colour,
                                           const PhiloxKeys& rk, uint32_t thr0, uint32_t thr1, uint64_t a1[4],
                                           uint64_t a0[4])
{
    if (!valid) item = 0;
    item_masks_lanes<F, ROUNDS>(g, item, q, t, colour, rk, thr0, thr1, a1, a0);
}

// One half-sweep of colour C over one lattice: block (x, y) owns items
// blockDim.x x .. of strip y (a 1-D block of 32 to 256 threads).  The draws
// need launch operands only (t from the host), so with programmatic dependent
// launch they run before the wait for the previous half-sweep, and fill the
// SMs that its last blocks leave idle; the lattice is read after it.  64
// registers keep 32 warps on an SM.  Bound by the issue of Philox products,
// XORs and compares (see accept_insert).  ROUNDS: Philox rounds of the draws
// (10, or the opt-in 7).
template <int C, bool UPDATE, bool RECORD, int ROUNDS = 10>
__global__ void __launch_bounds__(256, 4)
half_sweep_kernel(uint64_t* own, const uint64_t* other, Geom g, Strips st, SweepArgs a)
{
    __shared__ uint2 tab[kFields * kStripWords];
    pdl_launch();
    const uint32_t w0 = blockIdx.y * st.width;
    const bool last = blockIdx.y == st.n - 1u;
    const uint32_t width = last ? st.last : st.width;
    const uint32_t magic = last ? st.magic_last : st.magic;
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t grp = strip_group(q, magic);
    const uint32_t x = q - grp * width;
    const bool valid = grp * 4u < (uint32_t)g.L;
    uint32_t anti = 0, up = 0;
    ItemMasks acc;
    if (UPDATE) {
        const uint64_t t = sweep_number(a);
        first_products<kFields, kStripWords>(tab, w0, width, magic, philox_first_key((uint32_t)t, a.rk));
        if (valid) {
            const FirstTable first = {tab + x};
            draw_item<ROUNDS>(first, grp, t, C, a.rk, a.thr0, a.thr1, a.all0, a.all1, acc);
        }
    }
    pdl_wait();
    if (valid) apply_item<C, UPDATE, RECORD>(own, other, g, grp, w0 + x, acc, anti, up);
    if (RECORD) {
        const int slot = (blockIdx.x + gridDim.x * blockIdx.y) % kCountSlots;
        block_add_counts(record_counts(a) + 2 * slot, anti, up);
    }
}

}  // namespace ising
