// 2D stage launches: variant 0 = one thread per site, 1 = halo-tiled kernel,
// 2 / 3 = tiled / per site with the exact-sum stencil (FP64 only).
#include "stage_generic.cuh"
#include "stage_split.cuh"
#include "stage_tiled.cuh"

namespace nlse {

template <class T, int D, int ORDER>
cudaError_t launch_stage(const StageArgs<T>& A, const LaunchCfg& L, cudaStream_t stream) {
  constexpr bool fp64 = std::is_same<typename T::R, double>::value;
  const int variant = (!fp64 && L.variant >= 2) ? L.variant - 2 : L.variant;   // exact sums are FP64 only
  const bool exact = variant >= 2;
  const bool periodic = A.f.bc == BC_PERIODIC;
  // (the FP32 forms' tiled steps are step2d.cu's, small FP64 planes' exact-sum steps step2x.cu's; here their one thread
  // per site, and nlse_rhs, which takes the tiles on large periodic planes: F of 1500x1700 FP32 2SHOC 17 against 27 us,
  // of 128^2 4.2 by either)
  const bool tiles32 = !fp64 && variant == 1 && periodic && A.stage == 0 && (int64_t)A.f.n[0] * A.f.n[1] > 400000;
  if ((!fp64 && !tiles32) || variant == 0 || variant == 3 || (exact && A.f.fine)) {
    if (periodic) {
      if constexpr (fp64) if (exact) return launch_generic_periodic<T, D, ORDER, true>(A, stream);
      return launch_generic_periodic<T, D, ORDER>(A, stream);
    }
    if constexpr (fp64) if (exact) return launch_split<T, D, ORDER, true>(A, stream, true, true);
    return launch_split<T, D, ORDER>(A, stream, true, true);
  }
  // tiled: deep interior + the wall shell (periodic grids: the two layers at each end of each axis)
  auto deep = [&](cudaStream_t st) -> cudaError_t {
    if constexpr (fp64) if (exact) return launch2d_tiled<T, ORDER, true>(A, L.tile_cfg, st);
    return launch2d_tiled<T, ORDER>(A, L.tile_cfg, st);
  };
  auto shell = [&](cudaStream_t st) -> cudaError_t {
    if (periodic) {
      if constexpr (fp64) if (exact) return launch_shell_periodic<T, D, ORDER, true>(A, st);
      return launch_shell_periodic<T, D, ORDER>(A, st);
    }
    if constexpr (fp64) {
      if (exact) return launch_split<T, D, ORDER, true>(A, st, false, false);
      return launch_split<T, D, ORDER>(A, st, false, false);
    }
    return cudaErrorInvalidValue;
  };
  return launch_deep_and_shell(L, stream, has_deep(D, A.f.m), deep, shell);
}

#define INST(T, O) template cudaError_t launch_stage<T, 2, O>(const StageArgs<T>&, const LaunchCfg&, cudaStream_t);
INST(P64, 2) INST(P64, 4) INST(P32, 2) INST(P32, 4) INST(PMix, 2) INST(PMix, 4)
#undef INST

}  // namespace nlse
