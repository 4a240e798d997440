// Launchers of the paper's column-interleaved layout (ising_interleaved.cu).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "ising_device.cuh"

namespace ising {

bool ci_valid_side(int32_t L);   // L % 84 == 0 (N = L / 21 divisible by 4), 84 <= L <= 32760
cudaError_t ci_init_hot(uint64_t* S, int L, uint64_t seed, cudaStream_t s);
cudaError_t ci_init_cold(uint64_t* S, int L, int up, cudaStream_t s);
cudaError_t ci_pack(uint64_t* S, int L, const int8_t* spins, cudaStream_t s);
cudaError_t ci_unpack(const uint64_t* S, int L, int8_t* spins, cudaStream_t s);
// colour 0 does not record; in_graphs as for launch_half_sweep (ising_internal.h).
cudaError_t ci_half_sweep(int colour, bool update, bool record, uint64_t* S, int L, const SweepArgs& a,
                          bool in_graphs, cudaStream_t s);
// The paper's random-word chain (Sec. 4-5, Appendix A): iteration
// *a.t_base + a.t_off, phase 0 (the left floor(NC/2) columns of each of the
// nstrips strips of NC = L / nstrips columns) then phase 1 (the rest), one
// block per strip; thresholds and round keys from `a` (always 10 Philox
// rounds).  With `draws` (ci_rw_draw_bytes(L, nstrips) bytes of device
// memory; used when ci_rw_predraw(L, nstrips)) the updates' draws are made
// first on all SMs; with nullptr each block draws its own.
bool ci_valid_strips(int32_t L, int32_t nstrips);   // nstrips divides L, L / nstrips >= 2
size_t ci_rw_draw_bytes(int L, int nstrips);
// The lattice to and from the dense array of the cluster path (cl_dense_bytes
// in ising_internal.h): rows of one bit per spin, both colours.  ci_to_dense
// comes directly after a plain launch that triggers its dependents and writes
// neither array; it runs beside that launch and ends after it.  ci_from_dense
// also advances *t_dev (if not null) by n, and with `beside` its blocks are placed
// while the launch before, which triggers its dependents, runs.
cudaError_t ci_to_dense(const uint64_t* S, int L, uint32_t* dense, cudaStream_t s);
cudaError_t ci_from_dense(uint64_t* S, int L, const uint32_t* dense, uint64_t* t_dev, int64_t n, bool beside,
                          cudaStream_t s);
bool ci_rw_predraw(int L, int nstrips);
cudaError_t ci_random_words_iteration(uint64_t* S, int L, int nstrips, const SweepArgs& a, ulonglong2* draws,
                                      cudaStream_t s);
// The same with the updates planned ahead (ising_words.cu), where a half strip
// fits (words_planned): words_plan makes the plans of iterations
// sweep_number(a) .. + iterations - 1 (words_plan_bytes each; a buffer of
// words_buffer_bytes holds `iterations` of them, or ci_rw_draw_bytes, for any
// number of strips; words_most_iterations is as many as pay), words_run both phases of
// the plan's iteration `iteration` (0: right after words_plan, or after the
// phases before it); *err = 1 when a wait gave up; the first `stalls` (0 .. 2)
// phases wait for what never comes (a test hook).
bool words_planned(int L, int nstrips);
size_t words_plan_bytes(int L, int nstrips);
size_t words_buffer_bytes(int L, int iterations);
int words_most_iterations(int L);
cudaError_t words_plan(int L, int nstrips, const SweepArgs& a, int iterations, void* plan, cudaStream_t s);
cudaError_t words_run(uint64_t* S, int L, int nstrips, const void* plan, int iteration, unsigned int* err,
                      int stalls, cudaStream_t s);

}  // namespace ising
