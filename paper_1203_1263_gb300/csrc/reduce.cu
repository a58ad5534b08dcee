// FP64 reductions: mass, energy and max|V|.
//
// Each thread adds its terms exactly on the integer pipe (wide_sum.cuh) over its
// block's contiguous share of the sites, a block's threads are combined as
// integers, every block writes one (sum, compensation) pair, and the last block
// to finish adds the block pairs in a fixed order, so a result depends only on
// the input, never on scheduling.
//
// The energy's Laplacian is summed in 64-bit fixed point too, at a scale taken
// from the site's own operands, one per component; the sites next to a wall
// take the FP64 form, enumerated apart so that whole warps take it.  256^3 FP64
// state with V, mass and energy together: 655 us; with FP64 sums throughout
// (about 10 and 70 FP64 instructions per site) 3,180.  What bounds them now: the
// mass the FP64 pipe (79 % busy with the two instructions a site's |Psi|^2
// takes), the energy the FP64 pipe and the issue of the 26 conversions per site
// together (62 % and 45 % busy).
#include "nlse_device.cuh"
#include "nlse_internal.h"
#include "stage_generic.cuh"
#include "wide_sum.cuh"

namespace nlse {

// The block's pair into partials; the last block to get there adds all pairs and writes scale x the total, NaN if a
// block's sum left the FP64 range (the terms themselves are finite).  `done` counts the blocks (0 before and after).
__device__ __forceinline__ void finish(WideSum w, double* partials, unsigned int* done, double scale, double* result) {
  __shared__ bool last;
  w = block_wide_sum<256>(w);
  if (threadIdx.x == 0) {
    double s, c;
    w.pair(&s, &c);
    __stcg(partials + 2 * blockIdx.x, s);
    __stcg(partials + 2 * blockIdx.x + 1, c);
    __threadfence();
    last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  WideSum t;
  bool ok = true;
  for (int i = threadIdx.x; i < 2 * (int)gridDim.x; i += 256) {
    const double x = *(volatile const double*)(partials + i);
    if (finite_bits(x)) t.add(x);
    else ok = false;
  }
  ok = __syncthreads_and(ok);
  t = block_wide_sum<256>(t);
  if (threadIdx.x == 0) {
    double s, c;
    t.pair(&s, &c);
    result[0] = ok ? scale * (s + c) : __longlong_as_double(0x7FF8000000000000ll);
    *done = 0u;
  }
}

// The contiguous share [lo, hi) of a block, a multiple of its 256 threads.
__device__ __forceinline__ void block_share(int64_t total, int64_t* lo, int64_t* hi) {
  const int64_t per = ((total + gridDim.x - 1) / gridDim.x + 255) / 256 * 256;
  *lo = min((int64_t)blockIdx.x * per, total);
  *hi = min(*lo + per, total);
}

__device__ __forceinline__ void mass_term(WideSum& t, bool& bad, double2 p) {
  const double m2 = norm2(p);
  const bool ok = finite_bits(m2);
  bad |= !ok;
  if (ok) t.add(m2);
}
__device__ __forceinline__ void mass_term(WideSum& t, bool& bad, float2 p) {
  const bool ok = finite_bits(p.x) && finite_bits(p.y);
  bad |= !ok;
  if (ok) {
    t.add_square(p.x);
    t.add_square(p.y);
  }
}

template <class C>
__global__ void __launch_bounds__(256) k_mass(const C* __restrict__ psi, int64_t total, double* partials,
                                              unsigned int* flag, unsigned int* done, double scale, double* result) {
  WideSum t;
  bool bad = false;
  int64_t lo, hi;
  block_share(total, &lo, &hi);
  constexpr int U = 4;   // loads of a thread in flight
  for (int64_t i0 = lo + threadIdx.x; i0 < hi; i0 += U * 256) {
    C p[U];
#pragma unroll
    for (int u = 0; u < U; ++u) p[u] = i0 + u * 256 < hi ? __ldg(psi + i0 + u * 256) : C{0, 0};
#pragma unroll
    for (int u = 0; u < U; ++u) mass_term(t, bad, p[u]);
  }
  if (bad) atomicOr(flag, 2u);
  finish(t, partials, done, scale, result);
}

// One component of the stencil sum 16 s1 - s2 - 30 d Psi_c (order 2: s1 - 2 d Psi_c) of operands v[0] (the
// centre) and v[1 ..] (2 d nearest, then 2 d second neighbours), summed exactly in fixed point with the
// largest operand below 2^55 (see the bounds at fix1); NaN if an operand is not finite.
template <int D, int ORDER>
__device__ __forceinline__ double stencil_sum(const double* v) {
  constexpr int N = ORDER == 4 ? 4 * D + 1 : 2 * D + 1;
  unsigned int E = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) E = max(E, expo_bits(v[i]));
  if (E == 2047u) return __longlong_as_double(0x7FF8000000000000ll);
  const int F = 1077 - int(E);
  long long s1 = 0, s2 = 0;
#pragma unroll
  for (int i = 1; i <= 2 * D; ++i) s1 += fix1(v[i], F);
  if constexpr (ORDER == 2) return i2d_rn(s1 - 2 * D * fix1(v[0], F), -F);
#pragma unroll
  for (int i = 2 * D + 1; i < N; ++i) s2 += fix1(v[i], F);
  return i2d_rn(16 * s1 - s2 - 30 * D * fix1(v[0], F), -F);
}

// a Lap Psi at a site none of whose operands lies beyond a wall.
template <class T, int D, int ORDER, class Acc>
__device__ __forceinline__ double2 energy_lap(const Field<T>& f, const Acc& acc, double2 pc) {
  constexpr int N = ORDER == 4 ? 4 * D + 1 : 2 * D + 1;
  double x[N], y[N];
  x[0] = pc.x;
  y[0] = pc.y;
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int q = 0; q < (ORDER == 4 ? 4 : 2); ++q) {
      const double2 u = acc.at1(k, q == 0 ? -1 : (q == 1 ? 1 : (q == 2 ? -2 : 2)));
      const int i = q < 2 ? 1 + 2 * k + q : 1 + 2 * D + 2 * k + (q - 2);
      x[i] = u.x;
      y[i] = u.y;
    }
  return {f.cL * stencil_sum<D, ORDER>(x), f.cL * stencil_sum<D, ORDER>(y)};
}

// I: index type of the site decodes (64-bit divisions are long sequences).  P: periodic, every site counts and
// neighbours wrap; otherwise the interior sites: with 2SHOC first those two or more cells from every wall (`deep`
// of them, from index 2 on), then the `shell` next to the walls.
template <class T, int D, int ORDER, class I, bool P>
__global__ void __launch_bounds__(256, 3) k_energy(const Field<T> f, int64_t deep, int64_t shell, double* partials,
                                                unsigned int* flag, unsigned int* done, double scale, double* result) {
  constexpr bool SHELL = ORDER == 4 && !P;
  WideSum t;
  bool bad = false;
  auto add = [&](double2 pc, double m2, double v, double2 aL) {
    const double e = fma(-0.5 * f.s, m2 * m2, fma(v, m2, -fma(pc.x, aL.x, pc.y * aL.y)));
    const bool ok = finite_bits(e);
    bad |= !ok;
    if (ok) t.add(e);
  };
  int64_t lo, hi;
  block_share(deep, &lo, &hi);
  for (int64_t i = lo + threadIdx.x; i < hi; i += 256) {
    int idx[D];
    I rem = I(i);
    int64_t c = 0;
#pragma unroll
    for (int k = D - 1; k >= 0; --k) {
      const I mk = I(P ? f.n[k] : (SHELL ? f.n[k] - 4 : f.m[k])), q = rem / mk;
      idx[k] = int(rem - q * mk) + (P ? 0 : (SHELL ? 2 : 1));
      rem = q;
      c += idx[k] * f.st[k];
    }
    const double2 pc = ld2<double>(f.in, c);
    double2 aL;
    if constexpr (P) aL = energy_lap<T, D, ORDER>(f, GAccP<T, D>(f, c, idx), pc);
    else aL = energy_lap<T, D, ORDER>(f, GAcc<T, D>(f, c), pc);
    add(pc, norm2(pc), ldv<double>(f.V, c), aL);
  }
  if constexpr (SHELL) {
    block_share(shell, &lo, &hi);
    for (int64_t i = lo + threadIdx.x; i < hi; i += 256) {
      int idx[D];
      const int64_t c = shell_decode<T, D, I>(f, I(i), idx);
      const double2 pc = ld2<double>(f.in, c);
      const double m2 = norm2(pc), v = ldv<double>(f.V, c);
      add(pc, m2, v, a_lap_wall<T, D, ORDER>(f, GAcc<T, D>(f, c), idx, c, pc, fma(f.s, m2, -v)));
    }
  }
  if (bad) atomicOr(flag, 2u);
  finish(t, partials, done, scale, result);
}

template <class VR>
__global__ void __launch_bounds__(256) k_vmax(const VR* __restrict__ V, int64_t total, unsigned long long* out) {
  double m = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs(double(V[i])));
  // non-negative doubles order like their bit patterns
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// Largest range_bits over the components of a complex128 array into *out
// (exact-sum scale of the current state; *out must start at 0).
__global__ void __launch_bounds__(256) k_max_expo(const double* __restrict__ v, int64_t n, unsigned int* out) {
  unsigned int e = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    e = max(e, range_bits(__ldg(v + i)));
  emax_commit(out, e);
}

// Fraction bits of the exact-sum stencil for the state whose largest range_bits
// is E (collected in *emax by k_max_expo or by stage 4): F = 1077 - E.  A zero
// state keeps F0; a non-finite one keeps the previous F (the non-finite flag
// reports it).  `offset` is a test hook (nlse_debug_set).  Resets *emax for the
// next step.
__global__ void k_fix_update(unsigned int* emax, int* fdev, int F0, int offset) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const unsigned int E = *emax;
    if (E == 0u) *fdev = F0 + offset;
    else if (E < 2047u) *fdev = 1077 - int(E) + offset;
    *emax = 0u;
  }
}

cudaError_t launch_max_expo(const double* psi, int64_t n, unsigned int* expo, cudaStream_t stream) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  k_max_expo<<<(unsigned)b, 256, 0, stream>>>(psi, n, expo);
  return cudaGetLastError();
}

cudaError_t launch_fix_update(const double* psi, int64_t n, unsigned int* emax, int* fdev, int F0, int offset,
                              cudaStream_t stream) {
  if (psi) {
    const cudaError_t e = launch_max_expo(psi, n, emax, stream);
    if (e != cudaSuccess) return e;
  }
  k_fix_update<<<1, 32, 0, stream>>>(emax, fdev, F0, offset);
  return cudaGetLastError();
}

// One site per thread up to six blocks per SM (a small grid's reduction is latency), then more each: one wave of
// the mass kernel, two of the energy's (three blocks per SM).
constexpr int kReduceBlocks = 6 * 152;
static_assert(kReduceBlocks <= kMaxReduceBlocks, "a pair of partials per block");
static_assert((int64_t(1) << 40) / kReduceBlocks + 1024 < (int64_t(1) << 31), "a block's terms of the largest grid (wide_sum.cuh)");
static int reduce_blocks(int64_t work) {
  int64_t b = (work + 255) / 256;
  if (b < 1) b = 1;
  if (b > kReduceBlocks) b = kReduceBlocks;
  return int(b);
}

cudaError_t launch_mass(const void* psi, bool psi_double, int64_t total, double scale, double* partials,
                        double* result, unsigned int* flag, unsigned int* done, cudaStream_t stream) {
  const int nb = reduce_blocks(total);
  if (psi_double)
    k_mass<double2><<<nb, 256, 0, stream>>>((const double2*)psi, total, partials, flag, done, scale, result);
  else
    k_mass<float2><<<nb, 256, 0, stream>>>((const float2*)psi, total, partials, flag, done, scale, result);
  return cudaGetLastError();
}

template <class T, int D, int ORDER>
cudaError_t launch_energy(const Field<T>& f, double scale, double* partials, double* result, unsigned int* flag,
                          unsigned int* done, cudaStream_t stream) {
  const bool periodic = f.bc == BC_PERIODIC;
  int64_t deep = 1, shell = 0;
  for (int k = 0; k < D; ++k) deep *= periodic ? f.n[k] : (ORDER == 4 ? (f.n[k] > 4 ? f.n[k] - 4 : 0) : f.m[k]);
  if (!periodic && ORDER == 4) shell = f.ninterior - deep;
  const int nb = reduce_blocks(deep > shell ? deep : shell);
  auto run = [&](auto kern) {
    kern<<<nb, 256, 0, stream>>>(f, deep, shell, partials, flag, done, scale, result);
    return cudaGetLastError();
  };
  const bool small = f.ninterior < (int64_t(1) << 31) && deep < (int64_t(1) << 31);
  if (periodic) return small ? run(k_energy<T, D, ORDER, uint32_t, true>) : run(k_energy<T, D, ORDER, uint64_t, true>);
  return small ? run(k_energy<T, D, ORDER, uint32_t, false>) : run(k_energy<T, D, ORDER, uint64_t, false>);
}

#define INST(T, D, O) \
  template cudaError_t launch_energy<T, D, O>(const Field<T>&, double, double*, double*, unsigned int*, unsigned int*, \
                                             cudaStream_t);
INST(P64, 1, 2) INST(P64, 1, 4) INST(P64, 2, 2) INST(P64, 2, 4) INST(P64, 3, 2) INST(P64, 3, 4)
INST(E32, 1, 2) INST(E32, 1, 4) INST(E32, 2, 2) INST(E32, 2, 4) INST(E32, 3, 2) INST(E32, 3, 4)
INST(EMix, 1, 2) INST(EMix, 1, 4) INST(EMix, 2, 2) INST(EMix, 2, 4) INST(EMix, 3, 2) INST(EMix, 3, 4)
#undef INST

cudaError_t launch_vmax(const void* V, bool v_double, int64_t total, unsigned long long* out, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), stream);
  if (e != cudaSuccess) return e;
  const int nb = reduce_blocks(total);
  if (v_double) k_vmax<double><<<nb, 256, 0, stream>>>((const double*)V, total, out);
  else k_vmax<float><<<nb, 256, 0, stream>>>((const float*)V, total, out);
  return cudaGetLastError();
}

}  // namespace nlse
