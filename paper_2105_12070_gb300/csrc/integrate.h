// Internal interface between the host side of the library (chem_kernels.cu) and the integrate
// kernels, which are compiled in one translation unit per cell-group width G (integrate_g*.cu)
// so that the build runs in parallel.  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "chem_internal.h"

// Threads per CTA of the integrate kernels that keep two matrices per cell (8 warps: with ~250 registers per
// thread that is the register file, and shared memory holds 4 cells of 53 species)
#ifndef CHEM_MAX_THREADS_PER_CTA
#define CHEM_MAX_THREADS_PER_CTA 256
#endif

namespace chemgpu {

// Arguments of one integrate launch (all pointers device memory).
struct IntegrateArgs {
  double p, dt, rtol, atol;
  double *T, *Y;
  double* h_inout;
  int32_t* status;
  int32_t* steps_out;
  int32_t* rej_out;
  unsigned long long* totals;  // steps, rejects, failed cells, refine fallbacks
  int* queue;
  int64_t ncells;     // number of cells in the arrays (the stride of Y)
  int64_t first;      // this launch integrates cells first .. first + count - 1
  int64_t count;
  int max_steps;
  int use_queue;
  int mixed;          // 0: FP64 factors; 1: FP32 factors, 2: FP32 pairs (+ FP64-residual refinement)
  int refine_sweeps;  // refinement sweeps per stage solve (mixed)
  double* rec;        // record mode: checkpoint of every accepted step (NULL: off)
  int rec_cap;        // checkpoints per cell
  int solver;         // CHEM_SOLVER_*
  int fdjac;          // forward-difference Jacobian instead of the analytical one
  const double* p_cells;  // per-cell pressure in Pa (NULL: p for every cell)
  unsigned long long* phase;  // per-phase cycle counters (builds with CHEM_PHASE_TIMERS; else NULL)
};
// The kernels of one group width: the Rosenbrock solve with the analytical Jacobian and FP64 factors (the
// default, and the only one that records), Seulex, and the Rosenbrock solve with every option
// (low-precision factors, forward-difference Jacobian), whose code would cost the default registers.
enum : int { kIntegrateFp64 = 0, kIntegrateSeulex = 1, kIntegrateOptions = 2 };
inline int integrate_variant(int solver, bool mixed, bool fdjac) {
  return solver != 0 ? kIntegrateSeulex : (mixed || fdjac) ? kIntegrateOptions : kIntegrateFp64;
}

// Resident CTAs per SM the kernels are compiled for.  Groups of one warp serve small mechanisms, whose
// cells take a few KB of shared memory: there the registers limit the warps per SM, and two CTAs of
// 128 registers a thread hide more latency than one of 255.
constexpr int integrate_min_ctas(int G) { return G == 1 ? 2 : 1; }

// Threads per CTA of a variant: the default's compact plan puts five cells of 53 species on an SM, 10 warps
// of 2 per cell at 168 registers a thread (three warps on two of the four sub-partitions).
// Shear layer of 6080 cells: 2454 -> 2784 cells/s against four cells at 244 registers.  2432 cells, ms with 320
// and with 256 threads: 40 species / 200 reactions 167 and 180, 53 / 325 415 and 463; where only four cells
// fit an SM the smaller register budget costs nothing: 58 / 330 904 and 905, 60 / 360 1409 and 1405, 62 / 390
// 890 and 893.
constexpr int integrate_max_threads(int G, int variant) {
  return (G == 2 && variant == kIntegrateFp64) ? CHEM_MAX_THREADS_PER_CTA / 4 * 5 : CHEM_MAX_THREADS_PER_CTA;
}
// Which plan of a cell (make_plan) a variant works on.
constexpr int integrate_plan(int variant) { return variant == kIntegrateFp64 ? 1 /* kPlanCompact */ : 0 /* kPlanFull */; }

// The integrate kernel of one group width (G = 1, 2, 4 or 8 warps per cell) and variant, for occupancy
// queries and attributes; NULL for another G.
const void* integrate_kernel_fn(int G, int variant);

// Launches it: grid CTAs of `threads` threads with `smem` bytes of dynamic shared memory each,
// the per-cell plan of make_plan(K, R, n_pd, G).
void integrate_launch(int G, int variant, int grid, int threads, size_t smem, cudaStream_t st, const DevMech& d,
                      const IntegrateArgs& a);

// One translation unit per G defines these.
const void* integrate_kernel_fn_g1(int variant);
const void* integrate_kernel_fn_g2(int variant);
const void* integrate_kernel_fn_g4(int variant);
const void* integrate_kernel_fn_g8(int variant);
void integrate_launch_g1(int variant, int grid, int threads, size_t smem, cudaStream_t st, const DevMech& d,
                         const IntegrateArgs& a);
void integrate_launch_g2(int variant, int grid, int threads, size_t smem, cudaStream_t st, const DevMech& d,
                         const IntegrateArgs& a);
void integrate_launch_g4(int variant, int grid, int threads, size_t smem, cudaStream_t st, const DevMech& d,
                         const IntegrateArgs& a);
void integrate_launch_g8(int variant, int grid, int threads, size_t smem, cudaStream_t st, const DevMech& d,
                         const IntegrateArgs& a);

}  // namespace chemgpu
