// Launches of the 1D several-steps kernel (stage_step1d.cuh) and the choice of its tile.
#include "stage_step1d.cuh"
#include "nlse_internal.h"

namespace nlse {

// CTAs of `own` sites for an n-site line, and the end of CTA b's own sites.  Between walls the last site goes with
// the one before it: a boundary site's F reaches one site further inwards than its neighbour's, so it needs that
// neighbour owned too.
inline int line_ctas(int n, int own, bool periodic) { return ((periodic ? n : n - 1) + own - 1) / own; }
__device__ __forceinline__ int own_end(int b, int own, int n, bool periodic) {
  const int e = (b + 1) * own;
  return e >= (periodic ? n : n - 1) ? n : e;
}

template <class T, int ORDER, int NT, int SPT>
__global__ void __launch_bounds__(NT + 32) k_steps1d(const __grid_constant__ Step1Args<T> A, int halo, int steps) {
  using S = Steps1<T, ORDER, NT, SPT>;
  using C = typename T::C;
  __shared__ __align__(16) C buf[2 * S::W];
  const bool periodic = A.bc == BC_PERIODIC;
  const int own = S::RW - 2 * halo, tid = threadIdx.x;
  S t{A, buf, (int)blockIdx.x * own - halo, (int)blockIdx.x * own, own_end((int)blockIdx.x, own, A.n, periodic), tid >= NT, -1};
  // no wall within reach of any of the CTA's sites: no wall logic
  const bool walls = !(periodic || (t.x0 >= 2 && t.x0 + S::RW <= A.n - 2));
  if (t.wall_warp && walls) {   // lanes 0..3: sites 0, 1, n - 2, n - 1 (n == 3: 0, 1, -, 2), where the CTA has them
    const int l = tid - NT, g = l < 2 ? l : (l < 4 ? A.n - 4 + l : -1);
    const int c = min(max(g, 1), A.n - 2);   // F is evaluated there
    if (g >= t.x0 && g < t.x0 + S::RW && c >= t.x0 && c < t.x0 + S::RW && g >= 0 && !(l == 2 && g < 2)) t.site = g;
  }
  // the thread's sites: q-th slot
  auto slot = [&](int q) { return t.wall_warp ? t.site - t.x0 : tid + q * NT; };
  auto mine = [&](int q) { return t.wall_warp ? (q == 0 && t.site >= 0) : true; };
  auto inner = [&](int g) { return !walls || t.wall_warp || (g >= 2 && g <= A.n - 3); };   // else the wall warp's
  grid_launch_dependents();
#pragma unroll
  for (int q = 0; q < SPT; ++q) {   // V is no output of an earlier launch
    const int g = t.x0 + slot(q);
    const int c = periodic ? t.wrap(g) : min(max(g, 1), A.n - 2);
    t.v[q] = A.V && mine(q) ? typename T::R(__ldg(A.V + c)) : typename T::R(0);
  }
  if (tid < 4) {
    const int e = tid < 2 ? tid : S::RW + tid;
    buf[e] = buf[S::W + e] = C{0, 0};
  }
  grid_wait();
#pragma unroll
  for (int q = 0; q < SPT; ++q) {
    const int j = slot(q), g = t.x0 + j;
    const int w = periodic ? t.wrap(g) : g;
    t.m[q] = mine(q) && w >= 0 && w < A.n ? A.in[w] : typename T::M{0, 0};
    if (mine(q) && inner(g)) buf[j + 2] = stage_value<T>(t.m[q]);
  }
  __syncthreads();
  if (walls) t.template run<true>(steps);
  else t.template run<false>(steps);
#pragma unroll
  for (int q = 0; q < SPT; ++q) {
    const int g = t.x0 + slot(q);
    if (mine(q) && inner(g) && g >= t.own_lo && g < t.own_hi) A.out[g] = t.m[q];
  }
}

template <int ORDER, int SITES>
__global__ void __launch_bounds__(2 * SITES + 32) k_steps1d_split(const __grid_constant__ Step1Args<P64> A, int halo,
                                                                  int steps) {
  using S = Split1<ORDER, SITES>;
  __shared__ __align__(16) double buf[4 * S::W];
  const bool periodic = A.bc == BC_PERIODIC;
  const int own = SITES - 2 * halo, tid = threadIdx.x;
  S t{A, buf, (int)blockIdx.x * own - halo, (int)blockIdx.x * own, own_end((int)blockIdx.x, own, A.n, periodic),
      tid >= 2 * SITES, tid / 2, tid & 1};
  const bool walls = !(periodic || (t.x0 >= 2 && t.x0 + SITES <= A.n - 2));
  bool mine = true;
  if (t.wall_warp) {   // as in k_steps1d, a lane pair per site
    const int l = tid / 2 - SITES, g = l < 2 ? l : (l < 4 ? A.n - 4 + l : -1), c = min(max(g, 1), A.n - 2);
    const bool here = walls && g >= 0 && !(l == 2 && g < 2) && g >= t.x0 && g < t.x0 + SITES && c >= t.x0 && c < t.x0 + SITES;
    t.slot = here ? g - t.x0 : -1;
    mine = here;
  } else if (walls) {
    const int g = t.x0 + t.slot;
    mine = g >= 2 && g <= A.n - 3;
  }
  const int g = t.x0 + t.slot, w = periodic ? t.wrap(g) : g, c = periodic ? w : min(max(g, 1), A.n - 2);
  grid_launch_dependents();
  t.v = A.V && mine ? __ldg(A.V + c) : 0.0;
  if (tid < 8) {
    const int e = tid < 4 ? tid : 2 * (SITES + 2) + tid - 4;
    buf[e] = buf[2 * S::W + e] = 0.0;
  }
  grid_wait();
  const double* in = reinterpret_cast<const double*>(A.in);
  t.m = mine ? in[2 * (int64_t)w + 1 - t.k] : 0.0;
  if (mine) buf[2 * (t.slot + 2) + 1 - t.k] = t.m;
  __syncthreads();
  if (walls) t.template run<true>(steps);
  else t.template run<false>(steps);
  if (mine && g >= t.own_lo && g < t.own_hi) reinterpret_cast<double*>(A.out)[2 * (int64_t)g + 1 - t.k] = t.m;
}

namespace {

template <class K, class T>
cudaError_t launch_shape(K kern, int sites, int threads, const Step1Args<T>& A, int halo, int steps, bool early, cudaStream_t stream) {
  const int own = sites - 2 * halo;
  return launch_early(early, kern, dim3((unsigned)line_ctas(A.n, own, A.bc == BC_PERIODIC)), dim3((unsigned)threads + 32), 0,
                      stream, A, halo, steps);
}

// The sites per CTA and the most steps per launch (a power of two up to 8) of an n-site line.
struct Plan { int sites, steps; };

// FP64: the least estimate of 17 FP64 instructions of 64 cycles for every warp of a sub-partition and stage, times
// the CTAs per SM (not rounded up: launches overlap), and a launch's 2,600 cycles shared by its steps.  us per step
// with MSD walls: 2001 sites 8.6 (48 sites x 2 steps; 112 x 2 10.7), 10,000 12.0 (112 x 2; 48 x 1 13.4), 20,000 14.6
// (112 x 1; 112 x 2 16.8).  Wider CTAs never won: 240 x 1 at 32,000 sites 22.3 against 18.6.
Plan plan64(int n) {
  Plan best = {48, 2};
  double least = -1.0;
  for (int sites : {48, 112})
    for (int steps : {1, 2, 4}) {
      const int own = sites - 16 * steps;
      if (own < 16) continue;
      const double ctas = double(line_ctas(n, own, true)), per_sm = ctas > 152.0 ? ctas / 152.0 : 1.0;
      const double cost = 4.0 * per_sm * ((2 * sites + 32) / 128) * 17 * 64 + 2600.0 / steps;
      if (least < 0.0 || cost < least) {
        least = cost;
        best = {sites, steps};
      }
    }
  return best;
}

// FP32 stages: eight steps of 256 sites while those fill the chip once; beyond, a smaller share of halo (us per step:
// 5,000 sites 1.83 with 256 x 8 and 1.95 with 256 x 4; 100,000: 2.59 and 2.28, mixed form 512 x 8 5.29 and 256 x 4
// 7.71; 3e6: 1024 x 2 20.0 and 256 x 4 22.1, mixed 68 and 84).
Plan plan32(int n, bool mixed) {
  if (n <= 152 * 128) return {256, 8};
  if (n <= 200000) return mixed ? Plan{512, 8} : Plan{256, 4};
  return {1024, 2};
}

template <int ORDER>
cudaError_t launch_order(const Step1Args<P64>& A, int steps, bool early, cudaStream_t stream) {
  const Plan p = plan64(A.n);
  const int halo = 8 * p.steps;
  switch (p.sites) {
    case 48: return launch_shape(k_steps1d_split<ORDER, 48>, 48, 96, A, halo, steps, early, stream);
    default: return launch_shape(k_steps1d_split<ORDER, 112>, 112, 224, A, halo, steps, early, stream);
  }
}
template <int ORDER, class T>
cudaError_t launch_order(const Step1Args<T>& A, int steps, bool early, cudaStream_t stream) {
  const Plan p = plan32(A.n, !std::is_same<T, P32>::value);
  const int halo = 8 * p.steps;
  switch (p.sites) {
    case 256: return launch_shape(k_steps1d<T, ORDER, 256, 1>, 256, 256, A, halo, steps, early, stream);
    case 512: return launch_shape(k_steps1d<T, ORDER, 256, 2>, 512, 256, A, halo, steps, early, stream);
    default: return launch_shape(k_steps1d<T, ORDER, 256, 4>, 1024, 256, A, halo, steps, early, stream);
  }
}

}  // namespace

template <class T>
int steps1d_per_launch(int n) {
  if (std::is_same<T, P64>::value) return plan64(n).steps;
  return plan32(n, !std::is_same<T, P32>::value).steps;
}

template <class T>
cudaError_t launch_steps1d(const Step1Args<T>& A, int order, int steps, bool early, cudaStream_t stream) {
  return order == 4 ? launch_order<4>(A, steps, early, stream) : launch_order<2>(A, steps, early, stream);
}

#define INST(T)                                                                              \
  template int steps1d_per_launch<T>(int);                                                   \
  template cudaError_t launch_steps1d<T>(const Step1Args<T>&, int, int, bool, cudaStream_t);
INST(P64) INST(P32) INST(PMix)
#undef INST

}  // namespace nlse
