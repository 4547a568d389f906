// aap_kernels.cuh -- host-callable launchers of the step kernels.
#pragma once

#include <cuda_runtime.h>

#include "aap_internal.cuh"

namespace aapk {

// Everything one step launch needs; the step index and buffer parity are read
// on the device from Ctl, so a captured CUDA graph of steps can be replayed.
struct LaunchCfg {
    Sys *sys;                    // device array [nsys]
    int nsys;
    int model;                   // shared by all systems of the launch
    const int *tile_base;        // device [nsys + 1]: prefix of tiles per system
    Ctl *ctl;
    unsigned char *scratch;      // device [grid_step * scratch_per_block]
    size_t scratch_per_block;
    int scratch_cap;             // particles a block can stage in global scratch
    int spill_list_cap;          // spill matches a block can hold
    int threads;                 // 256 or 512
    int stage_cap;               // particles staged in shared memory
    int nce_max;                 // cells of the largest tile plus its ring
    int hist_words;              // histogram bins (theta + |Omega|) of the widest system
    int grid_step, grid_finish;
    // pipelined step (pipe_species: systems of several species): shared buffers of pipe_cap
    // staged / pipe_cap_own own particles per tile, one block per SM; tiles
    // that do not fit go to dense_list (device [job_count], zero between steps)
    int pipe, pipe_species;
    int pipe_few;                // at most kFewPerBlock tiles per block: a job list is kept (k_tile_order)
    int pipe_jobs;               // ... and claimed from; else tiles in raster order
    int pipe_cap, pipe_cap_own, pipe_grid;
    int pipe_nceh;               // half cells (split along x) of the largest extended tile, (2 tw + 4)(th + 2)
    int *dense_list;
    int2 *jobs;                  // device [job_bytes(job_tiles)]: what is claimed, in order (k_tile_order)
    int job_tiles;
    // many steps per launch (a small system, one block per tile, all resident)
    int multi, multi_species, multi_cap, multi_tiles, multi_threads;
    int multi_slices;            // scratch slices its tiles share
    int *multi_cnt;              // device: three private counter sets, two barrier words and a lock per slice, zero
                                 // between launches
    // metric-free step (knn > 0): cell count, scan, scatter, k-nearest update
    int knn;
    long long mf_n, mf_ncell;
    int mf_grid;                 // persistent blocks of the k-nearest update
};

// The pipelined step's jobs: up to one per tile and kMaxParts more, the tiles'
// costs (scratch), and {leading jobs for whole blocks, jobs, whether the order
// matters}.
constexpr int kMaxParts = 1024;
// Up to 12 tiles per SM a list is kept.  Of uneven states, with the list / in raster
// order, us per step: VM at 10 tiles per SM 126 / 144, at 13 153 / 167, at 18 214 / 217, at
// 23 254 / 257, at 28 289 / 280; NVM at 13 132 / 155, at 18 170 / 192; Langevin at 20 151 /
// 151.  So the gain ends between 23 and 28; the line is older than the check for
// even states, which lost at any number, and lies on the safe side.
constexpr int kFewPerBlock = 12;
inline size_t job_count(int tiles) { return (size_t)tiles + kMaxParts; }
inline size_t job_bytes(int tiles) { return job_count(tiles) * sizeof(int2) + (size_t)round_up(tiles, 4) * 4 + 16; }
inline float *job_cost(const LaunchCfg &L) { return reinterpret_cast<float *>(L.jobs + job_count(L.job_tiles)); }
inline int *job_meta(const LaunchCfg &L) { return reinterpret_cast<int *>(job_cost(L) + round_up(L.job_tiles, 4)); }

size_t step_smem_bytes(int stage_cap, int nce_max, int hist_words);
// Set the dynamic shared-memory limit of the step kernel and report how many
// of its blocks fit on one SM.
cudaError_t configure_step_kernel(int model, int threads, size_t smem_bytes, int *blocks_per_sm);

// Raw buffers of the pipelined step kernel: a tile's holds its staged records
// from the copy until its update is done (the update reads its own particles'
// records there).
#ifndef AAP_PIPE_RAW_BUFFERS
#define AAP_PIPE_RAW_BUFFERS 3
#endif
constexpr int kPipeRawBuffers = AAP_PIPE_RAW_BUFFERS;

// Dynamic shared memory of the pipelined step kernel; nceh: half cells of the
// largest extended tile, (2 tw + 4)(th + 2).
__host__ __device__ inline size_t pipe_smem_bytes(int cap, int cap_own, int nceh, int hist_words)
{
    return (size_t)(kPipeRawBuffers + 2) * cap * 16 + 2 * (size_t)round_up(nceh + 1, 8) * 2 +
           4 * (size_t)round_up(cap_own, 8) * 2 + 2 * (size_t)round_up(2 * cap, 8) * 2 +
           (size_t)round_up(nceh, 4) * 4 + (size_t)(kMaxTile + 4) * 4 + 2 * (size_t)round_up(hist_words, 4) * 4;
}
// Static shared memory of the pipelined step kernel of a model; its dynamic
// limit; the test hook of its waits (the wait bound, <= 0: default, and the
// stall injection).  The _species functions are those of the kernel for
// several species.
cudaError_t pipe_static_smem(int model, size_t *bytes);
cudaError_t configure_pipe_kernel(int model, size_t smem);
cudaError_t set_pipe_test(long long wait_cycles, int stall);
cudaError_t pipe_static_smem_species(int model, size_t *bytes);
cudaError_t configure_pipe_kernel_species(int model, size_t smem);
cudaError_t set_pipe_test_species(long long wait_cycles, int stall);
cudaError_t launch_step_pipe_species(const LaunchCfg &L, cudaStream_t st);
// The pipelined step kernel alone (launch_step adds k_finish).
cudaError_t launch_step_pipe(const LaunchCfg &L, cudaStream_t st);

// Ints of one private counter set: a line per tile and one for the spill count.
inline int multi_stride(int ntiles) { return (ntiles + 1) * kCntStride; }
inline size_t multi_bytes(int ntiles) { return (3 * (size_t)multi_stride(ntiles) + 4 + ntiles) * sizeof(int); }
// Decide whether a system of ntiles tiles can run many steps per launch (L.multi): all its blocks resident with at
// least min_cap staged records each.
cudaError_t configure_multi(LaunchCfg &L, bool species, int ntiles, int sm_count, int min_cap);
cudaError_t launch_multi(const LaunchCfg &L, int nsteps, cudaStream_t st);
cudaError_t set_multi_test(long long wait_cycles, int stall);

// One full step: k_step (or the pipelined step kernel) then k_finish.  With ev != nullptr, ev[0..2] are
// recorded before k_step, after k_step and after k_finish.
cudaError_t launch_step(const LaunchCfg &L, cudaStream_t st, cudaEvent_t *ev = nullptr);

// Blocks of the metric-free update that are resident at once on sm_count SMs.
cudaError_t configure_mf_kernels(int model, int knn, int hist_words, int sm_count, int *grid);

// The metric-free step (knn > 0): the kernels of launch_step for a flat system.
cudaError_t launch_mf_step(const LaunchCfg &L, cudaStream_t st, cudaEvent_t *ev);

cudaError_t launch_insert(const Sys &S, int b, const double *x, const double *y, const float *th,
                          int mode, cudaStream_t st);
// The jobs of the pipelined step, in the order they are claimed, from the tiles' current loads.
cudaError_t launch_tile_order(const LaunchCfg &L, cudaStream_t st);
// Whether the order matters (the third word of job_meta) to host memory.
cudaError_t copy_dense(const LaunchCfg &L, int *dst, cudaStream_t st);
// The largest tile load and staged set of buffer b into S.err[1] and [2].
cudaError_t launch_tile_load(const Sys &S, int b, cudaStream_t st);
// bad[0]: the lowest index with a position outside [0, lx] x [0, ly]; bad[1]:
// the lowest with a non-finite orientation; ~0 where there is none.
cudaError_t launch_validate(const double *x, const double *y, const float *th, long long n, double lx, double ly,
                            unsigned long long *bad, cudaStream_t st);
cudaError_t launch_gather(const Sys &S, int b, double *x, double *y, float *th, int *seen,
                          cudaStream_t st);
cudaError_t launch_observe(const Sys &S, int b, unsigned long long *out, cudaStream_t st);
// Start a measurement window of `nsys` systems (device array) at their current states in buffer b.
cudaError_t launch_begin_measure(Sys *sys, int nsys, long long max_n, int b, unsigned long long *sums, long long until,
                                 cudaStream_t st);
// Coarse-grained fields of buffer b into out[3][nby][nbx] (device), using
// acc[3 * nbx * nby] (device scratch, zero before and after) for the integer sums.
cudaError_t launch_coarse(const Sys &S, int b, int nbx, int nby, unsigned long long *acc, float *out,
                          cudaStream_t st);

}  // namespace aapk
