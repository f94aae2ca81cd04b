// Host-side launchers of the library's kernels (internal interface between the
// C ABI in mp_api.cu and the kernel translation units).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

namespace mpk {

struct ReduceParams {
  const DevSystem* systems;
  const double* records;
  double* est;  // MP_NEST doubles per system
  int64_t n_therm, n_meas;
  // Sort space for the distribution coefficient of systems with more than
  // MP_R_MAX_PATHS paths: 2 n_paths doubles at 2 rec_offset per system
  // (nullptr when no system is that large).
  double* sort_buf;
  double* work;  // scratch of the reduction's passes, reduce_work_doubles() doubles
};

struct BackwardParams {
  const DevSystem* systems;
  const double* records;
  const double* g_e;
  const double* g_m;
  double* grad_beta;
  double* grad_h;
};

// Shared-memory sweep kernels.  `variant` selects the kernel: L > 0 a batch
// of simple cubic lattices of that one size, -1 open chains only, 0 a batch
// of uneven sizes (the kernel switches per work item).
bool sweep_supports_L(int precision, int L);
cudaError_t sweep_prepare(int precision, int variant, int device, int* max_dynamic,
                          int* max_threads);
cudaError_t sweep_occupancy(int precision, int variant, int cta, int smem, int* blocks_per_sm);
cudaError_t launch_sweep(int precision, int variant, const SweepParams& p, int grid, int cta,
                         int smem, cudaStream_t st);

// Open chains only, each with at least as many threads as sites of a colour.
constexpr int kChainOne = -6;
// The streamed kernels compiled for simple cubic L = 32 and L = 64 (all
// systems of the batch streamed at that size).
constexpr int kStreamL32 = -1032;
constexpr int kStreamL64 = -1064;

// The square-lattice Ising kernel (any even L, sizes mixed or not).
constexpr int kIsingKernel = -3;
struct IsingThreads {
  int full, loaded;
};
IsingThreads ising_threads(int L, int64_t paths_per_sm, int smem_max, int ring, int most);
cudaError_t ising_prepare(int device, int* max_dynamic, int* max_threads);
cudaError_t ising_occupancy(int cta, int smem, int* blocks);
cudaError_t launch_ising(const SweepParams& p, int grid, int cta, int smem, cudaStream_t st);
// Slice bytes of an Ising path: 16 thresholds (aligned to 128 bytes within
// their 256), then per colour one word for every x/2 and block of four rows,
// and a copy of the first block.
constexpr int kIsingThrBytes = 256;
constexpr int ising_slice_spin_bytes(int L) { return kIsingThrBytes + 2 * 4 * (L / 2) * ((L + 3) / 4 + 1); }

// The random-site order (MP_FLAG_RANDOM_SITE, variant kRandomSiteKernel): one
// warp per path (one thread for many paths of very few sites), lattices in shared
// memory, or in HBM
// (random_site_bytes_per_site bytes per site and path).
constexpr int kRandomSiteKernel = -4;
struct RandomSitePlan {
  bool shared = false, thread_per_path = false;
  int slice = 0, cta = 0, smem = 0, grid = 0;  // shared-memory bytes per warp, launch shape
};
int random_site_bytes_per_site(int precision);
cudaError_t random_site_plan(int precision, int64_t max_sites, int64_t total_paths, int device, RandomSitePlan* plan);
cudaError_t launch_random_site(int precision, const RandomSitePlan& plan, const SweepParams& p, int n_systems,
                               int64_t total_paths, void* lattice, int64_t elements, cudaStream_t st);

cudaError_t reduce_prepare();  // raise the dynamic shared memory limit
int64_t reduce_work_doubles(int64_t total_paths, int n_systems);
cudaError_t launch_reduce(const ReduceParams& p, int n_systems, int64_t max_paths, cudaStream_t st);
cudaError_t launch_backward(const BackwardParams& p, int n_systems, cudaStream_t st);
cudaError_t launch_philox(const uint32_t* ctr, int64_t n, uint64_t seed, uint32_t* out,
                          cudaStream_t st);

}  // namespace mpk
