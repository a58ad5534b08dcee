// Launches of the 2D FP64 whole-step kernel (stage_step2x.cuh) and the choice of its tile.
#include "stage_step2x.cuh"
#include "nlse_internal.h"

namespace nlse {

namespace {

constexpr int kTX = 16, kNT = 256, kPerSm = 2;   // 16 columns: two CTAs per SM, and enough of them on small grids

template <int ORDER>
__global__ void __launch_bounds__(kNT, kPerSm) k_step2x(const __grid_constant__ Step2xArgs A, int ty, int ntx) {
  extern __shared__ __align__(16) unsigned char step2x_smem_[];
  Step2xTile<ORDER, kTX, kNT> tile(A, ty, blockIdx.x % ntx, blockIdx.x / ntx, step2x_smem_);
  grid_launch_dependents();
  tile.load_potential();
  grid_wait();
  tile.run();
}

int tiles(int ny, int nx, bool periodic, int ty, int* ntx) {
  int nty;
  step2_tiles(ny, nx, periodic, kTX, ty, ntx, &nty);
  return *ntx * nty;
}

template <int ORDER>
cudaError_t launch_order(const Step2xArgs& A, int ty, int ntx, int n, bool early, cudaStream_t stream) {
  auto kern = k_step2x<ORDER>;
  static SmemLimit limit;
  const cudaError_t e = limit.allow(kern, 227 * 1024);
  if (e != cudaSuccess) return e;
  return launch_early(early, kern, dim3((unsigned)n), dim3(kNT), step2x_smem(kTX, ty, A.V != nullptr), stream, A, ty, ntx);
}

}  // namespace

// One wave of 16-row tiles (up to 273 x 273): beyond, the halo's FP64 work costs more than the stage kernels'
// launches (us per step, Dirichlet 2SHOC: 256^2 24.0 against 47.5; 450^2 55 against 48, periodic 54 against 37).
bool step2x_fits(int ny, int nx, bool periodic) {
  int ntx;
  return (int64_t)ny * nx < (int64_t(1) << 20) && tiles(ny, nx, periodic, 16, &ntx) <= kPerSm * 152;
}

cudaError_t launch_step2x(const Step2xArgs& A, int order, bool early, cudaStream_t stream) {
  // 8-row tiles while those are one wave too (128^2: 16.7 against 19.1 us)
  const bool periodic = A.bc == BC_PERIODIC;
  int ntx, ty = 8, n = tiles(A.n[0], A.n[1], periodic, ty, &ntx);
  if (n > kPerSm * 152) n = tiles(A.n[0], A.n[1], periodic, ty = 16, &ntx);
  return order == 4 ? launch_order<4>(A, ty, ntx, n, early, stream) : launch_order<2>(A, ty, ntx, n, early, stream);
}

}  // namespace nlse
