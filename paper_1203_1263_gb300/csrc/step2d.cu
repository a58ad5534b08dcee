// Single-run launches of the 2D whole-step kernel (stage_step2d.cuh) and the choice of its tile.
#include "stage_step2d.cuh"
#include "nlse_internal.h"

namespace nlse {

template <class T, int ORDER, int TX, int NT, int RY, int MINB, bool WRAP>
__global__ void __launch_bounds__(NT, MINB) k_step2d(const __grid_constant__ Step2Args<T> A, int ty, int ntx) {
  extern __shared__ __align__(16) unsigned char step2_smem[];
  Step2Tile<T, ORDER, TX, NT, RY, WRAP> tile(A, ty, blockIdx.x % ntx, blockIdx.x / ntx, step2_smem);
  // may start while the step before still runs: V is not its output, Psi^n is
  tile.load_potential();
  grid_wait();
  tile.run();
}

namespace {

// The shapes of tile_cfg 0..3: columns, threads, rows per strip, CTAs per SM that their registers allow.
struct Shape { int tx, nt, ry, per_sm; };
constexpr Shape kShapes[4] = {{32, 256, 2, 3}, {64, 256, 2, 3}, {32, 256, 4, 3}, {64, 384, 4, 2}};

// Rows of the tile of shape s for an ny x nx grid: those of the least estimated time (SM cycles).  A tile costs its
// latency (its loads and barriers, kLoad, and each round of strips through its threads) and its share of the
// SM's shared-memory rate (kSite per evaluated site); the grid costs whole waves of the former or the
// whole chip's rate of the latter, whichever is longer.  The constants are fitted to steps of 31^2 to
// 1732^2 grids over every shape and height (256^2: 8.6 us with 32 x 8 tiles, 9.3 with 32 x 16; 1000^2:
// 23.3 with 64 x 32, 25.3 with 64 x 24; 1732^2: 51 with 64 x 32, 60 with 64 x 16).
int plan(const Shape& s, int ny, int nx, bool periodic, bool with_v) {
  constexpr long long kLoad = 4000, kSms = 152, kSmem = 228 * 1024;
  long long best = -1;
  int ty_best = 4;
  for (int ty = 4; ty <= 64; ty += 4) {
    const size_t smem = s.tx == 32 ? step2_smem<32>(ty, with_v) : step2_smem<64>(ty, with_v);
    if (smem > 227 * 1024) break;
    int ntx, nty;
    step2_tiles(ny, nx, periodic, s.tx, ty, &ntx, &nty);
    const long long tiles = (long long)ntx * nty;
    long long res = kSmem / (long long)(smem + 1024);
    if (res > s.per_sm) res = s.per_sm;
    long long sites = 0, rounds = 0;
    for (int e = 6; e >= 0; e -= 2) {
      const long long n = (long long)(s.tx + 2 * e) * (ty + 2 * e);
      sites += n;
      rounds += (n / (2 * s.ry) + s.nt - 1) / s.nt;
    }
    const long long waves = (tiles + res * kSms - 1) / (res * kSms), per_sm = (tiles + kSms - 1) / kSms;
    const long long lat = waves * rounds * (500 + 375 * s.ry), rate = per_sm * sites * 3 / 4;
    const long long cost = waves * kLoad + (lat > rate ? lat : rate);
    if (best < 0 || cost < best) {
      best = cost;
      ty_best = ty;
    }
  }
  return ty_best;
}

// WRAP: a periodic grid's kernel (its wrapped loads cost the others 5 % in one kernel for both: 1000^2 FP32, MSD, central
// differences 16.9 against 16.1 us per step).
template <class T, int ORDER, int CFG, bool WRAP>
cudaError_t launch_wrap(const Step2Args<T>& A, int ty, bool early, cudaStream_t stream) {
  constexpr Shape s = kShapes[CFG];
  const size_t smem = step2_smem<s.tx>(ty, A.V != nullptr);
  auto kern = k_step2d<T, ORDER, s.tx, s.nt, s.ry, s.per_sm, WRAP>;
  static SmemLimit limit;
  const cudaError_t e = limit.allow(kern, 227 * 1024);
  if (e != cudaSuccess) return e;
  int ntx, nty;
  step2_tiles(A.n[0], A.n[1], WRAP, s.tx, ty, &ntx, &nty);
  return launch_early(early, kern, dim3((unsigned)(ntx * nty)), dim3(s.nt), smem, stream, A, ty, ntx);
}

template <class T, int ORDER, int CFG>
cudaError_t launch_shape(const Step2Args<T>& A, int ty, bool early, cudaStream_t stream) {
  return A.bc == BC_PERIODIC ? launch_wrap<T, ORDER, CFG, true>(A, ty, early, stream)
                             : launch_wrap<T, ORDER, CFG, false>(A, ty, early, stream);
}

template <class T, int ORDER>
cudaError_t launch_order(const Step2Args<T>& A, int tile_cfg, bool early, cudaStream_t stream) {
  // 64 columns (a smaller share of halo) where the grid fills the chip with them, 32 below: 400^2 9.3 against
  // 11.1 us per step, 600^2 12.9 against 12.1, 1300^2 32.5 against 30.2
  const int cfg = tile_cfg >= 0 ? tile_cfg : ((long long)A.n[0] * A.n[1] > 250000 ? 1 : 0);
  const int ty = plan(kShapes[cfg], A.n[0], A.n[1], A.bc == BC_PERIODIC, A.V != nullptr);
  switch (cfg) {
    case 0: return launch_shape<T, ORDER, 0>(A, ty, early, stream);
    case 1: return launch_shape<T, ORDER, 1>(A, ty, early, stream);
    case 2: return launch_shape<T, ORDER, 2>(A, ty, early, stream);
    default: return launch_shape<T, ORDER, 3>(A, ty, early, stream);
  }
}

}  // namespace

template <class T>
cudaError_t launch_step2d(const Step2Args<T>& A, int order, int tile_cfg, bool early, cudaStream_t stream) {
  return order == 4 ? launch_order<T, 4>(A, tile_cfg, early, stream) : launch_order<T, 2>(A, tile_cfg, early, stream);
}

template cudaError_t launch_step2d<P32>(const Step2Args<P32>&, int, int, bool, cudaStream_t);
template cudaError_t launch_step2d<PMix>(const Step2Args<PMix>&, int, int, bool, cudaStream_t);

}  // namespace nlse
