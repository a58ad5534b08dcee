// 3D stage launches: variant 0 = one thread per site, 1 = z-marching tiled kernel
// (TMA-fed when the layout allows, else cooperative loads; FP32 forms of a few
// million sites or without TMA: columns through the L1 cache),
// 2 / 3 = tiled / generic with the exact-sum stencil (FP64 only).
// Included by one small translation unit per (precision, order), so that the
// many kernel instantiations compile in parallel.
#pragma once
#include "stage_generic.cuh"
#include "stage_march.cuh"
#include "stage_pair.cuh"
#include "stage_slab.cuh"
#include "stage_split.cuh"
#include "stage_tiled.cuh"
#include "stage_tma.cuh"

namespace nlse {

template <class T, int D, int ORDER>
cudaError_t launch_stage(const StageArgs<T>& A, const LaunchCfg& L, cudaStream_t stream) {
  constexpr bool fp64 = std::is_same<typename T::R, double>::value;
  const int variant = (!fp64 && L.variant >= 2) ? L.variant - 2 : L.variant;   // exact sums are FP64 only
  const bool exact = variant >= 2;
  const bool periodic = A.f.bc == BC_PERIODIC;
  if (variant == 0 || variant == 3) {
    if (periodic) {
      if constexpr (fp64) if (exact) return launch_generic_periodic<T, D, ORDER, true>(A, stream);
      return launch_generic_periodic<T, D, ORDER>(A, stream);
    }
    if constexpr (fp64) if (exact) return launch_split<T, D, ORDER, true>(A, stream, true, true);
    if constexpr (std::is_same<T, P64>::value) {
      // see the figures in stage_pair.cuh, and walls_apart
      const int64_t sites = (int64_t)A.f.n[0] * A.f.n[1] * A.f.n[2];
      if (sites <= (ORDER == 4 ? 600000 : 16384) && walls_apart<T, D, ORDER, false>(A.f, true))
        return launch_pair<ORDER>(A, stream);
    }
    return launch_split<T, D, ORDER>(A, stream, true, true);
  }
  if constexpr (!fp64) {
    // one launch (the hook that drives the TMA kernels' bounded waits keeps those)
    if (A.stage >= 1 && !L.extra_tx && march_serves<ORDER>(A.f, L.tmap != nullptr)) return launch_march<T, ORDER>(A, stream);
  }
  // tiled: deep interior (TMA-fed when the layout allows) + the wall shell, as
  // shared-memory slabs (FP32 stages: three x layers per x wall) or, for thin
  // grids and periodic grids (whose shell wraps), the global-memory shell kernel
  const bool slabs = slab_ok(A.f.n) && !periodic;
  constexpr int nsx = fp64 ? 1 : 3;   // x-wall layers owned by the slab shell
  StageArgs<T> B = A;
  B.xwall = slabs ? nsx - 1 : 0;
  auto deep = [&](cudaStream_t st) -> cudaError_t {
    if constexpr (fp64) {
      if (exact) return L.tmap ? launch3d_tma<T, ORDER, true>(B, L, st) : launch3d_tiled<T, ORDER, true>(B, L.tile_cfg, st);
    }
    return L.tmap ? launch3d_tma<T, ORDER, false>(B, L, st) : launch3d_tiled<T, ORDER>(B, L.tile_cfg, st);
  };
  auto shell = [&](cudaStream_t st) -> cudaError_t {
    if (periodic) {
      if constexpr (fp64) if (exact) return launch_shell_periodic<T, D, ORDER, true>(B, st);
      return launch_shell_periodic<T, D, ORDER>(B, st);
    }
    if (slabs) {
      if constexpr (fp64) if (exact) return launch_shell_slabs<T, ORDER, true, nsx>(B, st, L.side_yx);
      return launch_shell_slabs<T, ORDER, false, nsx>(B, st, L.side_yx);
    }
    if constexpr (fp64) if (exact) return launch_split<T, D, ORDER, true>(B, st, false, false);
    return launch_split<T, D, ORDER>(B, st, false, false);
  };
  if (slabs) return launch_deep_and_shell(L, stream, has_deep(D, A.f.m), deep, shell);
  LaunchCfg L1 = L;   // one shell kernel: no use for the slabs' extra streams
  L1.side_yx[0] = L1.side_yx[1] = nullptr;
  return launch_deep_and_shell(L1, stream, has_deep(D, A.f.m), deep, shell);
}

}  // namespace nlse
