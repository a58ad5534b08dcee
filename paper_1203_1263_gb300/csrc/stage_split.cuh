// The wall-aware per-site stage as three kinds of threads.
//
// A site next to a wall takes a longer chain of instructions than one in the
// deep interior (ghosts with divisions, then the boundary sites it serves, each
// with its own loads and stores), and in a kernel with one thread per interior
// site every warp of a row holds both kinds, so each warp runs both chains one
// after the other.  On small grids that chain is the stage's time.  Here the
// deep sites, the sites next to a wall and the boundary sites are three ranges of
// blocks: warps hold one kind, and a boundary site has a thread of its own, which
// evaluates F at its interior neighbour once more (MSD; Eq. msd) instead of
// waiting for that site's thread (where that pays: walls_apart).  The arithmetic is site_rhs, serve_walls and
// rk_apply as everywhere, so results are bit-for-bit those of one thread per
// interior site (21^3 FP64 2SHOC MSD: 37.7 against 60.5 us per step; small FP64
// grids: stage_pair.cuh).  The kernel may start before the one before it has
// ended, so it reads what that wrote by ordinary loads (ld2_ordered).
#pragma once
#include "nlse_internal.h"
#include "stage_generic.cuh"

namespace nlse {

// The t-th boundary site: the sites with some index 0 or N - 1, as shell_decode's faces.
template <class T, int D, class I>
__device__ __forceinline__ int64_t boundary_decode(const Field<T>& f, I t, int* idx) {
  auto outer = [&](int k, int q) { return q == 0 ? 0 : f.n[k] - 1; };
  if constexpr (D == 1) {
    idx[0] = outer(0, int(t));
  } else if constexpr (D == 2) {
    const I F0 = I(2) * I(f.n[1]);
    if (t < F0) {
      idx[0] = outer(0, t < I(f.n[1]) ? 0 : 1);
      idx[1] = int(t < I(f.n[1]) ? t : t - I(f.n[1]));
    } else {
      t -= F0;
      idx[0] = 1 + int(t >> 1);
      idx[1] = outer(1, int(t & 1));
    }
  } else {
    const I plane = I(f.n[1]) * I(f.n[2]), F0 = I(2) * plane, F1 = I(f.m[0]) * I(2) * I(f.n[2]);
    if (t < F0) {
      idx[0] = outer(0, t < plane ? 0 : 1);
      const I r = t < plane ? t : t - plane;
      idx[1] = int(r / I(f.n[2]));
      idx[2] = int(r % I(f.n[2]));
    } else if (t < F0 + F1) {
      t -= F0;
      const I pa = I(2) * I(f.n[2]);
      idx[0] = 1 + int(t / pa);
      const I r = t % pa;
      idx[1] = outer(1, r < I(f.n[2]) ? 0 : 1);
      idx[2] = int(r < I(f.n[2]) ? r : r - I(f.n[2]));
    } else {
      t -= F0 + F1;
      const I pa = I(2) * I(f.m[1]);
      idx[0] = 1 + int(t / pa);
      const I r = t % pa;
      idx[1] = 1 + int(r >> 1);
      idx[2] = outer(2, int(r & 1));
    }
  }
  int64_t s = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) s += idx[k] * f.st[k];
  return s;
}

inline int64_t boundary_count(int D, const int* n, const int* m) {
  int64_t all = 1, inner = 1;
  for (int k = 0; k < D; ++k) {
    all *= n[k];
    inner *= m[k];
  }
  return all - inner;
}

// The t-th of n sites next to the walls, without the boundary sites it serves.
template <class T, int D, int ORDER, bool EXACT, class I, bool FINE = false>
__device__ __forceinline__ unsigned int shell_site(const StageArgs<T>& A, int64_t t, int64_t n) {
  if (t >= n) return 0u;
  int idx[D];
  const int64_t c = shell_decode<T, D, I>(A.f, I(t), idx);
  const GAcc<T, D, true, FINE> acc(A.f, c);
  const PointVals<T> p = load_point<T, -1, EXACT>(A, c, true);
  typename V2<typename T::R>::t pc;
  typename T::R m2w;
  return rk_apply<T>(A, c, site_rhs<T, D, ORDER, EXACT>(A.f, acc, idx, c, p.v, &pc, &m2w), p);
}

// The t-th of n boundary sites.
template <class T, int D, int ORDER, bool EXACT, class I, bool FINE = false>
__device__ __forceinline__ unsigned int boundary_site(const StageArgs<T>& A, int64_t t, int64_t n) {
  using R = typename T::R;
  using C2 = typename V2<R>::t;
  const Field<T>& f = A.f;
  if (t >= n) return 0u;
  int idx[D];
  const int64_t b = boundary_decode<T, D, I>(f, I(t), idx);
  const PointVals<T> p = load_point<T, -1, EXACT>(A, b, true);
  C2 Fb = {R(0), R(0)};
  if (f.bc == BC_MSD) {   // see serve_walls
    const C2 pb = ld2_ordered<R>(f.in, b);
    int64_t c = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      idx[k] = min(max(idx[k], 1), f.n[k] - 2);
      c += idx[k] * f.st[k];
    }
    const GAcc<T, D, true, FINE> acc(f, c);
    C2 pc;
    R m2w;
    const C2 F = site_rhs<T, D, ORDER, EXACT>(f, acc, idx, c, ldv<R>(EXACT ? A.Vs : f.V, c), &pc, &m2w);
    const R m2 = EXACT ? m2w : norm2(pc);
    R theta = R(0);
    if (EXACT ? m2 > R(0) : m2 > f.tiny) theta = fma(F.y, pc.x, -(F.x * pc.y)) / m2;
    Fb = {-theta * pb.y, theta * pb.x};
  } else if (f.bc == BC_L0) {
    const C2 pb = ld2_ordered<R>(f.in, b);
    const R Nb = fma(EXACT ? f.sG : f.s, norm2(pb), -p.v);
    Fb = {-Nb * pb.y, Nb * pb.x};
  }
  return rk_apply<T>(A, b, Fb, p);
}

// Blocks [0, b1): the n1 deep sites; [b1, b2): the n2 shell sites; the rest: the n3 boundary sites.  Three CTAs per SM
// for the exact sums on planes (at two, a little over two CTAs per SM take a whole wave more: 282^2 56.2 against 48.8 us
// per step, 1000^2 243 and 191), two with the correction's operands (unbounded, 256^2 66.9 against 52.4).  The others are
// left to the compiler (0; a bound of one makes it take up to 26 registers more).
template <class T, int D, int ORDER, bool EXACT, class I, bool FINE = false>
__global__ void __launch_bounds__(256, EXACT && D == 2 ? (FINE ? 2 : 3) : 0)
    k_stage_split(const StageArgs<T> A, unsigned b1, unsigned b2, int64_t n1, int64_t n2, int64_t n3) {
  using R = typename T::R;
  using C2 = typename V2<R>::t;
  const Field<T>& f = A.f;
  unsigned int ex = 0;
  grid_wait();
  if (blockIdx.x < b1) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n1) {
      int idx[D];
      I rem = I(t);
      int64_t c = 0;
#pragma unroll
      for (int k = D - 1; k >= 0; --k) {
        const I mk = I(f.n[k] - 4), q = rem / mk;
        idx[k] = int(rem - q * mk) + 2;
        rem = q;
        c += idx[k] * f.st[k];
      }
      const GAcc<T, D, true, FINE> acc(f, c);
      const PointVals<T> p = load_point<T, -1, EXACT>(A, c, true);
      const C2 pc = acc.at0();
      const R N = fma(EXACT ? f.sG : f.s, norm2(pc), -p.v);
      C2 aL;
      if constexpr (EXACT) aL = a_lap_exact_deep<T, D, ORDER>(f, acc, idx, c, pc, N);
      else aL = a_lap_body<T, D, ORDER, GAcc<T, D, true, FINE>, false>(f, acc, idx, c, pc, N);
      ex = rk_apply<T>(A, c, {-fma(N, pc.y, aL.y), fma(N, pc.x, aL.x)}, p);
    }
  } else if (blockIdx.x < b2) {
    ex = shell_site<T, D, ORDER, EXACT, I, FINE>(A, (int64_t)(blockIdx.x - b1) * blockDim.x + threadIdx.x, n2);
  } else {
    ex = boundary_site<T, D, ORDER, EXACT, I, FINE>(A, (int64_t)(blockIdx.x - b2) * blockDim.x + threadIdx.x, n3);
  }
  if (A.emax) emax_commit(A.emax, ex);
}

// Whether the boundary sites get threads of their own, in a launch of every site (deep) or of the walls alone.  With
// MSD walls such a thread evaluates its interior neighbour's F a second time: that pays while the walls are latency
// beside the rest, and costs once they are work for the whole chip.  us per step, 2SHOC, MSD, one thread per interior
// site and this form:
//   every site, FP64 stencil   12x5000 48 / 42, 5x6000 37 / 33, 64^3 282 / 173; 3x20000 40 / 61, 9x200x300 324 / 369
//   every site, exact sums     21^3 89 / 81, 46^3 129 / 99, 64^3 222 / 144; 33^3 85 / 95, 5x6000 48 / 59
//   walls, exact sums          500^2 59 / 57, 3x40x40 91 / 78; 60x4000 61 / 65, 12x5000 51 / 63, 6x300x300 202 / 287
//   walls, FP64 stencil, 3D    3x40x40 65 / 37, 3x100x100 64 / 54; 100x5x100 68 / 72, 6x300x300 331 / 434
//   FP32                       700x700x9 (every site) 400 / 329; 6x600x700 (walls) 131 / 145
// (central differences, whose F is cheaper, later: walls, exact sums 200x200x4 53 / 45, 6x300x300 112 / 118).  The other
// boundaries' sites are a few instructions, apart in all but the largest exact-sum shells (Dirichlet 6x200000 262 / 303,
// 3x300x400 159 / 128).  Planes of the FP64 stencil: the tiles' CTAs pile up on the SMs that short wall CTAs leave free,
// from 40,000 to 110,000 sites (Dirichlet 128^2 30 / 22, 256^2 47 / 48, 100x700 48 / 83, 282^2 48 / 61, 500^2 110 / 107).
template <class T, int D, int ORDER, bool EXACT>
inline bool walls_apart(const Field<T>& f, bool deep) {
  int64_t total = 1;
  bool has_tiles = true;
  for (int k = 0; k < D; ++k) {
    total *= f.n[k];
    has_tiles &= f.n[k] >= 5;
  }
  const int64_t n3 = boundary_count(D, f.n, f.m);
  const bool msd = f.bc == BC_MSD;
  if constexpr (!std::is_same<typename T::R, double>::value) return !msd || n3 <= (deep && D == 3 ? total : 300000);
  if (deep) {
    if (!msd) return true;
    if (EXACT) return n3 <= (ORDER == 4 ? 1500 : 600000) || n3 * (D == 2 ? 16 : 8) <= total;
    return n3 <= 24000 || n3 * (D == 2 ? 16 : 10) <= total;
  }
  if (EXACT) {
    if (!msd) return n3 <= (D == 2 ? 100000 : 250000);
    return n3 <= (ORDER == 4 ? 3500 : (D == 2 ? 16000 : 100000));
  }
  if (D == 2 && has_tiles && total > 32768) return false;
  return !msd || n3 <= (has_tiles && ORDER == 4 && D == 3 ? 4000 : 24000);
}

// Every site (deep: the tiled kernels' part left out).  `early`: on the step's own stream, where the kernel before may
// still run.
template <class T, int D, int ORDER, bool EXACT = false>
cudaError_t launch_split(const StageArgs<T>& A, cudaStream_t stream, bool deep, bool early) {
  if (!walls_apart<T, D, ORDER, EXACT>(A.f, deep))
    return deep ? launch_generic<T, D, ORDER, EXACT>(A, stream) : launch_shell<T, D, ORDER, EXACT>(A, stream);
  int64_t n1 = 1;
  for (int k = 0; k < D; ++k) n1 *= A.f.n[k] > 4 ? A.f.n[k] - 4 : 0;
  const int64_t n2 = A.f.ninterior - n1, n3 = boundary_count(D, A.f.n, A.f.m);
  if (!deep) n1 = 0;
  const int threads = site_kernel_threads(n1 + n2 + n3);
  auto blocks = [&](int64_t n) { return (unsigned)((n + threads - 1) / threads); };
  const unsigned b1 = blocks(n1), b2 = b1 + blocks(n2), b3 = b2 + blocks(n3);
  auto run = [&](auto kern) -> cudaError_t {
    return launch_early(early, kern, dim3(b3), dim3((unsigned)threads), 0, stream, A, b1, b2, n1, n2, n3);
  };
  if constexpr (D == 2 && EXACT) {   // fine planes are small
    if (A.f.fine) return run(k_stage_split<T, D, ORDER, EXACT, uint32_t, true>);
  }
  if (A.f.ninterior + n3 < (int64_t(1) << 31)) return run(k_stage_split<T, D, ORDER, EXACT, uint32_t>);
  return run(k_stage_split<T, D, ORDER, EXACT, uint64_t>);
}

}  // namespace nlse
