// Launchers shared between the library's translation units (not exported).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "nlse_device.cuh"
#include "smem_limit.h"
#include "stage_step1d.cuh"
#include "stage_step2d.cuh"
#include "stage_step2x.cuh"

namespace nlse {

constexpr int kMaxReduceBlocks = 1024;

// A kernel that may start while the kernel before it in the stream still runs (programmatic dependent
// launch): it calls grid_wait() before it touches anything an earlier kernel wrote or still reads, and
// grid_launch_dependents() where the next kernel may start (otherwise as its CTAs end).  The early start pays
// where a CTA fills an SM or CTAs are many; where a grid is less than a wave of small CTAs, the next
// kernel's pile up on the SMs that are done first (64^3 FP32 columns 26.7 against 21.1 us per step without, 46^3
// one thread per site 20.2 and 16.6, 512^2 FP32 12.8 and 10.9; but 256^2 FP64 21.7 and 22.4, a batch 594
// and 602).  Before grid_wait() a kernel may read only what nobody writes while the call's kernels run (V, tables).  What
// wrote that before the call is ordered with it by an ordinary launch alone: the early start needs no more of the
// launch before than its CTAs' end, not that their stores are visible.  So the first launch of a call is an ordinary
// one (early = false; in a captured graph the first node has nothing before it).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... Q>
inline cudaError_t launch_early(bool early, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                Q&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// CTA tile (x-by-y threads) of the tiled 3D/2D kernels for tile_cfg 0..3.
inline void tma_tile_shape(int tile_cfg, int* tx, int* ty) {
  switch (tile_cfg) {
    case 1: *tx = 64; *ty = 4; break;
    case 2: *tx = 32; *ty = 16; break;
    case 3: *tx = 64; *ty = 8; break;
    default: *tx = 32; *ty = 8; break;
  }
}

// The FP32 form's fused step (two RK4 stages per pass; stage_fused.cuh): A[0..3]
// are stages 1..4, tm12 / tm34 the TMA descriptors of the passes' inputs
// (Psi^n, Psi_out) with the fused kernel's box (fused_box below).
template <int ORDER>
cudaError_t launch_fused_step(const StageArgs<P32>* A, const void* tm12, const void* tm34, const LaunchCfg& L,
                              cudaStream_t stream);
bool fused_grid_ok(int d, const int* n);
// the fused kernel's TMA box: 64 + 8 complex values by 8 + 8 rows
constexpr int kFusedBoxX = 2 * (64 + 8), kFusedBoxY = 8 + 8;

// One RK4 step of a 2D grid in one launch, Psi^n in A.in to Psi^{n+1} in A.out (stage_step2d.cuh).  early, here and
// below: not a call's first launch (launch_early).
template <class T>
cudaError_t launch_step2d(const Step2Args<T>& A, int order, int tile_cfg, bool early, cudaStream_t stream);

// The same for FP64 with the exact-sum stencil (stage_step2x.cuh); launch_max_expo puts the largest exponent of a
// complex128 array (n components) into the word of the first step.
bool step2x_fits(int ny, int nx, bool periodic);   // grids it is the faster one for
cudaError_t launch_step2x(const Step2xArgs& A, int order, bool early, cudaStream_t stream);
cudaError_t launch_max_expo(const double* psi, int64_t n, unsigned int* expo, cudaStream_t stream);

// Up to steps1d_per_launch(n) RK4 steps of an n-site line in one launch, from A.in to A.out (stage_step1d.cuh).
template <class T>
int steps1d_per_launch(int n);
template <class T>
cudaError_t launch_steps1d(const Step1Args<T>& A, int order, int steps, bool early, cudaStream_t stream);

// 1D lines on one thread-block cluster (stage_line1d.cuh): nsteps RK4 steps of
// an n-site line in one launch; A[0..3] are stages 1..4 with Psi updated in
// place.  cudaErrorInvalidConfiguration when the line does not fit or the
// cluster cannot be co-scheduled (the caller then takes the per-site kernel).
bool line_ok(int n);
cudaError_t launch_line_steps(const StageArgs<P64>* A, int64_t nsteps, int n, int order, int F0, int fix_offset,
                              cudaStream_t stream);

cudaError_t launch_mass(const void* psi, bool psi_double, int64_t total, double scale, double* partials,
                        double* result, unsigned int* flag, unsigned int* done, cudaStream_t stream);
template <class T, int D, int ORDER>
cudaError_t launch_energy(const Field<T>& f, double scale, double* partials, double* result, unsigned int* flag,
                          unsigned int* done, cudaStream_t stream);
cudaError_t launch_vmax(const void* V, bool v_double, int64_t total, unsigned long long* out, cudaStream_t stream);
// Exact-sum scale: with psi (complex128, n = 2 x sites components) first the
// largest exponent of psi into *emax, then *fdev = the fraction bits for it
// (+ offset) and *emax = 0.  With psi == nullptr only the second part (the
// exponent was collected by the stage-4 kernels).
cudaError_t launch_fix_update(const double* psi, int64_t n, unsigned int* emax, int* fdev, int F0, int offset,
                              cudaStream_t stream);
cudaError_t launch_round_master(const double2* master, float2* n32, int64_t total, cudaStream_t stream);
cudaError_t launch_scale_v(const double* V, double s, int64_t n, double* Vs, cudaStream_t stream);

}  // namespace nlse
