// The paper's random-word chain (Sec. 4-5, Appendix A) with its updates planned
// ahead.  A phase is one sequence of 10 N h word updates per strip, each on the
// word that its draws choose, and the result must be the sequential chain's,
// word for word.
//
// What bounds it: the longest chain of updates that touch one another (about
// 120 of the 3,360 of a half strip of 48 x 7 words).  ci_rw_phase_kernel finds
// the updates that may run in rounds of a window, six block barriers and a
// table of claims each: 82 us a phase at L = 1008 and 72 strips.  But which
// updates wait for which depends on the draws alone, not on the spins, so
// words_plan_kernel works it out beforehand on all SMs, for every phase and
// iteration of a call at once: each word's updates in sequence order, and with
// each the number of updates of its four neighbours that come before it.  In
// words_run_kernel a thread owns a word: it runs its next update as soon as the
// four neighbours have had exactly that many.  A word's spins (21 bits) and its
// count of updates share 64 bits of shared memory, so one load gives both and
// no barrier or fence is needed.  An update that is the oldest of all pending
// ones never waits, so the phase always ends.  Measured on GB300, 5 iterations
// of L = 1008 with 72 strips, a record after each: 798 -> 202 us, of which the
// plans take 54 and a phase 14.  (The plans of later iterations beside the
// phases, on a second stream: 218 against 215.)  A phase is bound by latency: 15%
// fewer instructions a look (the turns at the top and bottom rows in the warps that
// have them, four looks to a test for the end) gave 1 to 3%.
#include <cuda_runtime.h>

#include <algorithm>

#include "ising_device.cuh"
#include "ising_dense.cuh"
#include "ising_interleaved.cuh"
#include "ising_interleaved.h"
#include "ising_internal.h"
#include "ising_per_device.h"

namespace ising {
namespace {

constexpr int kPlanWarps = 8;
constexpr size_t kWordsSmemMax = 220 * 1024;
constexpr int kWordsThreads = 1024;             // most threads of a strip, one or two words each
constexpr int kWordsLooks = 4;                  // a thread's looks at its neighbours between two tests for the end
constexpr uint32_t kWordsTries = 1u << 22;      // such rounds of looks before it gives up
constexpr size_t kWordsPlanBytes = (size_t)64 << 20;      // of a handle's plans (at least one iteration's)
constexpr int kWordsPlanIterations = 16;
constexpr uint32_t kWordBits = (1u << 21) - 1;
constexpr int kWordIndexBits = 12;              // a half strip has at most 2 kWordsThreads words
static_assert(2 * kWordsThreads <= 1 << kWordIndexBits, "an update's word and four accept bits fit 16 bits");

// The strips' half strips in a phase.
struct WordsGeom {
    int L, N, NC, nstrips;
    __host__ __device__ int h(int phase) const { return phase == 0 ? NC / 2 : NC - NC / 2; }
    __host__ __device__ int words(int phase) const { return N * h(phase); }
    __host__ __device__ uint32_t updates(int phase) const { return 10u * (uint32_t)words(phase); }
    // plan of an iteration: entries of phase 0's strips, of phase 1's, then the starts
    __host__ __device__ size_t entry0(int phase, int strip) const
    {
        return phase == 0 ? (size_t)strip * updates(0) : (size_t)nstrips * updates(0) + (size_t)strip * updates(1);
    }
    __host__ __device__ size_t entries() const { return (size_t)nstrips * (updates(0) + updates(1)); }
    __host__ __device__ size_t start0(int phase, int strip) const
    {
        return phase == 0 ? (size_t)strip * (words(0) + 1)
                          : (size_t)nstrips * (words(0) + 1) + (size_t)strip * (words(1) + 1);
    }
    __host__ __device__ size_t starts() const { return (size_t)nstrips * (words(0) + words(1) + 2); }
    __host__ __device__ size_t bytes() const { return (entries() * sizeof(uint4) + starts() * 4 + 255) / 256 * 256; }
};

// An update as its word's thread needs it: x, y the accept masks r < thr1 and
// r < thr0 of its 21 spins, z the updates of the words above (low half) and
// below that come before it, w those of the words before and after in the row.
using Entry = uint4;

// Accept bits of spins K .. of a call's draws w[FROM .. 3] (spins 0 .. 20).
template <int K, int FROM>
__device__ __forceinline__ void words_accept(const uint32_t (&w)[4], const SweepArgs& a, uint32_t& m1, uint32_t& m0)
{
    if constexpr (FROM < 4 && K < 21) {
        accept_bit<K>(m1, w[FROM], a.thr1);
        accept_bit<K>(m0, w[FROM], a.thr0);
        words_accept<K + 1, FROM + 1>(w, a, m1, m0);
    }
}

// Calls B .. 5 of an update (the counter of call b is (step, 8 strip + b, t, x3),
// and draw 4 b + e is the word of spin 4 b + e - 2), with their first products.
template <int B>
__device__ __forceinline__ void words_calls(const PhiloxRowKey& row, const uint2 (&first)[6], const SweepArgs& a,
                                            uint32_t& m1, uint32_t& m0)
{
    if constexpr (B < 6) {
        uint32_t w[4];
        philox_row_tail<10>(row, a.rk, first[B].x, first[B].y, w);
        words_accept<4 * B - 2, 0>(w, a, m1, m0);
        words_calls<B + 1>(row, first, a, m1, m0);
    }
}

// The plan of strip blockIdx.x, phase blockIdx.y, iteration sweep_number(a) +
// blockIdx.z.  A warp takes a contiguous part of the sequence: first all count
// their parts' updates of each word, the counts become each part's first update
// numbers, then each goes through its part 32 updates at a time, with a table of
// the lanes that update a word.
__global__ void __launch_bounds__(32 * kPlanWarps)
words_plan_kernel(WordsGeom g, SweepArgs a, char* __restrict__ plan)
{
    extern __shared__ __align__(16) uint32_t plan_smem[];
    const int phase = blockIdx.y, strip = blockIdx.x, h = g.h(phase), W = g.words(phase);
    const uint32_t U = g.updates(phase);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* const cnt = plan_smem + (size_t)warp * W;                     // updates of a word before this warp's next
    uint32_t* const lanes = plan_smem + (size_t)(kPlanWarps + warp) * W;    // this chunk's lanes on a word
    uint32_t* const start = plan_smem + (size_t)2 * kPlanWarps * W;         // W + 1: first entries of the words
    uint16_t* const word = reinterpret_cast<uint16_t*>(start + W + 1);      // U: the updates' words, bits 0 and 1 of both masks
    plan += (size_t)blockIdx.z * g.bytes();
    Entry* const entry = reinterpret_cast<Entry*>(plan) + g.entry0(phase, strip);
    uint32_t* const starts = reinterpret_cast<uint32_t*>(plan + g.entries() * sizeof(Entry)) + g.start0(phase, strip);
    const uint64_t t = sweep_number(a) + blockIdx.z;
    const uint32_t x3 = 0x80000000u | ((uint32_t)(t >> 32) << 1) | (uint32_t)phase;
    const uint32_t part = (U + 32 * kPlanWarps - 1) / (32 * kPlanWarps) * 32;
    const uint32_t s0 = min(U, (uint32_t)warp * part), s1 = min(U, s0 + part);
    for (int i = threadIdx.x; i < 2 * kPlanWarps * W; i += blockDim.x) plan_smem[i] = 0;
    // the calls' first products, the same for every update of the strip
    const uint32_t key = philox_first_key((uint32_t)t, a.rk);
    uint2 first[6];
#pragma unroll
    for (int b = 0; b < 6; ++b) mul_hilo(kPhiloxM0, key ^ ((uint32_t)strip * 8u + b), first[b].x, first[b].y);
    __syncthreads();
    for (uint32_t s = s0 + lane; s < s1; s += 32) {
        uint32_t w[4], m1 = 0, m0 = 0;
        philox_row_tail<10>(philox_row_key(s, (uint32_t)t, x3, a.rk), a.rk, first[0].x, first[0].y, w);
        const uint32_t x = __umulhi(w[0], (uint32_t)g.N) * (uint32_t)h + __umulhi(w[1], (uint32_t)h);
        words_accept<0, 2>(w, a, m1, m0);
        word[s] = (uint16_t)(x | m1 << kWordIndexBits | m0 << (kWordIndexBits + 2));
        atomicAdd(cnt + x, 1u);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < W; x += blockDim.x) {
        uint32_t run = 0;
        for (int k = 0; k < kPlanWarps; ++k) {
            uint32_t* c = plan_smem + (size_t)k * W + x;
            const uint32_t v = *c;
            *c = run;
            run += v;
        }
        start[x] = run;
    }
    __syncthreads();
    if (warp == 0) {
        uint32_t before = 0;
        for (int x0 = 0; x0 < W; x0 += 32) {
            const uint32_t v = x0 + lane < W ? start[x0 + lane] : 0u;
            uint32_t sum = v;
            for (int d = 1; d < 32; d *= 2) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, sum, d);
                if (lane >= d) sum += o;
            }
            if (x0 + lane < W) start[x0 + lane] = before + sum - v;
            before += __shfl_sync(0xffffffffu, sum, 31);
        }
        if (lane == 0) start[W] = before;
    }
    __syncthreads();
    for (int x = threadIdx.x; x <= W; x += blockDim.x) starts[x] = start[x];
    for (uint32_t c0 = s0; c0 < s1; c0 += 32) {
        const uint32_t s = c0 + lane;
        const bool live = s < s1;
        const uint32_t kept = live ? word[s] : 0u, x = kept & ((1u << kWordIndexBits) - 1u);
        if (live) atomicOr(lanes + x, 1u << lane);
        __syncwarp();
        Entry e;
        uint32_t pos = 0, all = 0;
        if (live) {
            const uint32_t below = (1u << lane) - 1u, I = x / (uint32_t)h, j = x - I * (uint32_t)h;
            auto before = [&](uint32_t y) { return cnt[y] + __popc(lanes[y] & below); };
            const uint32_t up = I == 0 ? x + (uint32_t)(g.N - 1) * h : x - h;
            const uint32_t dn = I == (uint32_t)g.N - 1 ? j : x + h;
            e.z = before(up) | before(dn) << 16;
            e.w = (j > 0 ? before(x - 1) : 0u) | (j + 1 < (uint32_t)h ? before(x + 1) : 0u) << 16;
            pos = start[x] + before(x);
            all = lanes[x];
        }
        __syncwarp();
        if (live && lane == __ffs(all) - 1) {
            cnt[x] += __popc(all);
            lanes[x] = 0;
        }
        __syncwarp();
        if (!live) continue;
        uint32_t m1 = kept >> kWordIndexBits & 3u, m0 = kept >> (kWordIndexBits + 2);
        words_calls<1>(philox_row_key(s, (uint32_t)t, x3, a.rk), first, a, m1, m0);
        e.x = (m1 | a.all1) & kWordBits;
        e.y = (m0 | a.all0) & kWordBits;
#ifdef ISING_CHECKED
        if (!check_index(pos, U, __LINE__)) continue;
#endif
        entry[pos] = e;
    }
}

// The word at a shared address, one of the n at `win`.
__device__ __forceinline__ uint64_t word_look(uint32_t addr, uint32_t win, uint64_t n, uint32_t line)
{
    uint64_t v;
#ifdef ISING_CHECKED
    if (!check_index((addr - win) / 8u, n, line)) return 0;
#else
    (void)win;
    (void)n;
    (void)line;
#endif
    asm volatile("ld.volatile.shared.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}

// A word that a thread owns: its next update and where its neighbours are.
struct OwnWord {
    uint32_t at, up, dn;            // shared addresses of the word, of the words above and below
    bool first_row, last_row;
    uint32_t spins, done, count;
    uint32_t ahead;                 // shared address of the entry after `next`
    Entry e, next;                  // its next update and the one after
};

// The entry at a shared address, one of the n at `first`.
__device__ __forceinline__ Entry entry_ld(uint32_t addr, uint32_t first, uint32_t n, uint32_t line)
{
    Entry e;
#ifdef ISING_CHECKED
    if (!check_index((addr - first) / 16u, n, line)) return make_uint4(0, 0, 0, 0);
#else
    (void)first;
    (void)n;
    (void)line;
#endif
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(e.x), "=r"(e.y), "=r"(e.z), "=r"(e.w) : "r"(addr));
    return e;
}

// One phase of one iteration, strip blockIdx.x, from its plan.
template <int WPT>
__global__ void __launch_bounds__(kWordsThreads)
words_run_kernel(uint64_t* S, WordsGeom g, int phase, bool fresh, const char* __restrict__ plan, unsigned int* err,
                 uint32_t stall)
{
    extern __shared__ __align__(16) uint4 run_smem[];
    const int strip = blockIdx.x, h = g.h(phase), hw = h + 2, W = g.words(phase);
    const uint32_t U = g.updates(phase);
    const int col0 = strip * g.NC + (phase == 0 ? 0 : g.NC / 2);
    const uint64_t n_lat = (uint64_t)g.N * g.L;
    Entry* const entry = run_smem;                                          // U
    uint64_t* const win = reinterpret_cast<uint64_t*>(run_smem + U);        // N x (h + 2): spins | updates done << 32
    const uint64_t n_win = (uint64_t)g.N * hw;
    uint32_t* const start = reinterpret_cast<uint32_t*>(win + n_win);       // W + 1
    const Entry* const my_entry = reinterpret_cast<const Entry*>(plan) + g.entry0(phase, strip);
    const uint32_t* const my_start =
        reinterpret_cast<const uint32_t*>(plan + g.entries() * sizeof(Entry)) + g.start0(phase, strip);
    // the plan is of a launch that this one waits for (fresh), or one that ended
    // before the launch before passed its wait; the lattice is the launch before's
    if (fresh) pdl_wait();
    for (uint32_t i = threadIdx.x; i < U; i += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(entry + i)), "l"(my_entry + i) : "memory");
    for (int i = threadIdx.x; i <= W; i += blockDim.x) start[i] = __ldg(my_start + i);
    if (!fresh) pdl_wait();
    pdl_launch();
    for (int i = threadIdx.x; i < (int)n_win; i += blockDim.x) {
        const int I = i / hw;
        int J = col0 - 1 + i - I * hw;
        J = J < 0 ? J + g.L : (J >= g.L ? J - g.L : J);
        word_st(win, (uint64_t)i, pack_fields(word_ld<false>(S, (uint64_t)I * g.L + J, n_lat, __LINE__)), n_win,
                __LINE__);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const uint32_t win_sh = (uint32_t)__cvta_generic_to_shared(win), row = 8u * (uint32_t)hw;
    const uint32_t entry_sh = (uint32_t)__cvta_generic_to_shared(entry);
    OwnWord o[WPT];
#pragma unroll
    for (int k = 0; k < WPT; ++k) {
        // a thread without a word looks at word 0's neighbours and never runs
        const bool has = threadIdx.x + k * blockDim.x < (uint32_t)W;
        const int x = has ? threadIdx.x + k * blockDim.x : 0, I = x / h, j = x - I * h;
        o[k].first_row = I == 0;
        o[k].last_row = I == g.N - 1;
        o[k].at = win_sh + (uint32_t)I * row + 8u * (uint32_t)(j + 1);
        o[k].up = o[k].first_row ? o[k].at + (uint32_t)(g.N - 1) * row : o[k].at - row;
        o[k].dn = o[k].last_row ? o[k].at - (uint32_t)(g.N - 1) * row : o[k].at + row;
        o[k].spins = (uint32_t)word_look(o[k].at, win_sh, n_win, __LINE__);
        o[k].done = 0;
        o[k].count = has ? start[x + 1] - start[x] : 0u;
        // two entries past a word's last (never run) are other words', or the window's first bytes
        o[k].ahead = entry_sh + 16u * (start[x] + 2u);
        o[k].e = entry_ld(o[k].ahead - 32u, entry_sh, U + 2, __LINE__);
        o[k].next = entry_ld(o[k].ahead - 16u, entry_sh, U + 2, __LINE__);
        o[k].e.z |= stall;               // a test hook: a count that no word reaches
    }
    // rows whose neighbours come from across the top or bottom row: few warps have any
    bool edge = false;
#pragma unroll
    for (int k = 0; k < WPT; ++k) edge = edge || o[k].first_row || o[k].last_row;
    edge = __any_sync(0xffffffffu, edge);
    // a word changes by its own thread only, so there is no barrier from here on
    auto look = [&](OwnWord& w) {
        const uint64_t up = word_look(w.up, win_sh, n_win, __LINE__), dn = word_look(w.dn, win_sh, n_win, __LINE__);
        const uint64_t lf = word_look(w.at - 8, win_sh, n_win, __LINE__), rt = word_look(w.at + 8, win_sh, n_win, __LINE__);
        // the counts are below 2^16: at most 20,480 updates of a half strip
        const uint32_t z = (uint32_t)(up >> 32) | (uint32_t)(dn >> 32) << 16;
        const uint32_t v = (uint32_t)(lf >> 32) | (uint32_t)(rt >> 32) << 16;
        bool ready = w.done < w.count && z == w.e.z && v == w.e.w;
#ifdef ISING_CHECKED
        ready = ready && check_index((w.ahead - entry_sh) / 16u, U + 2, __LINE__);
#endif
        // straight-line: the lanes of a warp are seldom ready together
        uint32_t u = (uint32_t)up, d = (uint32_t)dn;
        if (edge) {
            u = w.first_row ? (u << 1 | u >> 20) & kWordBits : u;
            d = w.last_row ? (d >> 1 | d << 20) & kWordBits : d;
        }
        const uint32_t spins = flip_all(w.spins, u, d, (uint32_t)lf, (uint32_t)rt, w.e.x, w.e.y);
        w.spins = ready ? spins : w.spins;
        w.done += ready;
        w.ahead += ready ? 16u : 0u;
        w.e.x = ready ? w.next.x : w.e.x;
        w.e.y = ready ? w.next.y : w.e.y;
        w.e.z = ready ? w.next.z : w.e.z;
        w.e.w = ready ? w.next.w : w.e.w;
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
                     "@p st.volatile.shared.u64 [%5], %6;\n\t"
                     "@p ld.shared.v4.u32 {%0, %1, %2, %3}, [%7];\n\t}"
                     : "+r"(w.next.x), "+r"(w.next.y), "+r"(w.next.z), "+r"(w.next.w)
                     : "r"((uint32_t)ready), "r"(w.at), "l"((uint64_t)w.done << 32 | w.spins), "r"(w.ahead - 16u)
                     : "memory");
    };
    for (uint32_t tries = 0;; ++tries) {
        bool pending = false;
#pragma unroll
        for (int n = 0; n < kWordsLooks; ++n)
#pragma unroll
            for (int k = 0; k < WPT; ++k) look(o[k]);
#pragma unroll
        for (int k = 0; k < WPT; ++k) pending = pending || o[k].done < o[k].count;
        if (!__any_sync(0xffffffffu, pending)) break;
        if (tries == kWordsTries) {
            *(volatile unsigned int*)err = 1;
            break;
        }
    }
#pragma unroll
    for (int k = 0; k < WPT; ++k) {
        const int x = threadIdx.x + k * blockDim.x;
        if (x >= W) continue;
        const int I = x / h;
        word_st(S, (uint64_t)I * g.L + col0 + x - I * h, spread_fields(o[k].spins), n_lat, __LINE__);
    }
}

WordsGeom words_geom(int L, int nstrips) { return {L, L / 21, L / nstrips, nstrips}; }

size_t plan_smem_bytes(const WordsGeom& g)
{
    const size_t W = g.words(1);
    return (2 * kPlanWarps * W + W + 1) * 4 + ((size_t)g.updates(1) * 2 + 3) / 4 * 4;
}

size_t run_smem_bytes(const WordsGeom& g, int phase)
{
    return g.updates(phase) * sizeof(Entry) + (size_t)g.N * (g.h(phase) + 2) * 8 + ((size_t)g.words(phase) + 1) * 4;
}

bool words_setup()
{
    static PerDevice<bool> ok;
    return ok.get([] {
        constexpr auto kSmem = cudaFuncAttributeMaxDynamicSharedMemorySize;
        return cudaFuncSetAttribute(words_plan_kernel, kSmem, (int)kWordsSmemMax) == cudaSuccess &&
               cudaFuncSetAttribute(words_run_kernel<1>, kSmem, (int)kWordsSmemMax) == cudaSuccess &&
               cudaFuncSetAttribute(words_run_kernel<2>, kSmem, (int)kWordsSmemMax) == cudaSuccess;
    });
}

}  // namespace

bool words_planned(int L, int nstrips)
{
    const WordsGeom g = words_geom(L, nstrips);
    return g.words(1) <= 2 * kWordsThreads && run_smem_bytes(g, 1) <= kWordsSmemMax &&
           plan_smem_bytes(g) <= kWordsSmemMax && words_setup();
}

size_t words_plan_bytes(int L, int nstrips) { return words_geom(L, nstrips).bytes(); }

// The starts of any number of strips come to at most N L + L.
size_t words_buffer_bytes(int L, int iterations)
{
    const size_t NL = (size_t)(L / 21) * L;
    return (size_t)iterations * ((10 * NL * sizeof(Entry) + (NL + L) * 4 + 255) / 256 * 256);
}

int words_most_iterations(int L)
{
    return (int)std::max<size_t>(1, std::min<size_t>(kWordsPlanBytes / words_buffer_bytes(L, 1), kWordsPlanIterations));
}

cudaError_t words_plan(int L, int nstrips, const SweepArgs& a, int iterations, void* plan, cudaStream_t s)
{
    const WordsGeom g = words_geom(L, nstrips);
    words_plan_kernel<<<dim3(nstrips, 2, iterations), 32 * kPlanWarps, plan_smem_bytes(g), s>>>(
        g, a, static_cast<char*>(plan));
    return cudaGetLastError();
}

cudaError_t words_run(uint64_t* S, int L, int nstrips, const void* plan, int iteration, unsigned int* err,
                      int stalls, cudaStream_t s)
{
    const dim3 grid(nstrips);
    const WordsGeom g = words_geom(L, nstrips);
    const char* p = static_cast<const char*>(plan) + (size_t)iteration * g.bytes();
    for (int phase = 0; phase < 2; ++phase) {
        const int W = g.words(phase), per = W > kWordsThreads ? 2 : 1, threads = ((W + per - 1) / per + 31) / 32 * 32;
        const bool fresh = iteration == 0 && phase == 0;      // the plan is the launch before
        launch_pdl_with(false, run_smem_bytes(g, phase), per == 1 ? words_run_kernel<1> : words_run_kernel<2>, grid,
                        dim3(threads), s, S, g, phase, fresh, p, err, phase < stalls ? 0x8000u : 0u);
    }
    return cudaGetLastError();
}

}  // namespace ising
