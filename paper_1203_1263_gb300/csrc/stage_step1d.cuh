// Several RK4 steps of a 1D line in one launch.
//
// A line's step is a chain of four short stages, so launches, barriers between
// SMs and trips through memory are most of its time.  Here a CTA takes NT x SPT
// consecutive sites, `halo` of them on either side beyond the ones it owns,
// through `steps` whole steps on its own: every stage evaluates all its sites
// from the stage before in shared memory, after which two more sites at either
// edge hold values of no meaning, so with halo >= 8 steps the owned sites are
// right at the end.  Psi^n, K_tot and V of a site stay in its thread's
// registers; a stage is one CTA barrier.  The evaluated sites beyond the owned
// ones are the price; what bounds a step is the stages' dependent instructions
// (short lines) or the FP32 / FP64 rate (long ones), not memory: Psi is read and
// written once per launch.  Psi at the end goes to another buffer than at the
// start, because neighbouring CTAs still read that.
//
// The sites of the CTAs next to a wall that need wall code (the boundary sites
// and the interior sites beside them) belong to four lanes of one more warp, so
// that their longer chains (ghosts, the MSD wall's divisions) run beside the
// other sites' and not after them in the same warp: 2001 sites, FP64, Dirichlet
// walls, 8.5 us per step with the wall sites as a branch, 6.4 apart (4.6 on the
// periodic line).  A boundary site's lane evaluates F at its interior neighbour
// once more.  Every site's arithmetic is the per-site kernels' (site_rhs,
// rk_apply) in the same order, so results are bit-for-bit theirs.
#pragma once
#include "nlse_device.cuh"
#include "stage_step2d.cuh"

namespace nlse {

// T: P64, P32 or PMix.
template <class T>
struct Step1Args {
  using R = typename T::R;
  int n;
  int bc;
  R s, h2_over_a, cL, tiny;     // as in Field
  R dtc[4];                     // dt/2, dt/2, dt, dt/6
  const typename T::VR* V;      // or nullptr
  const typename T::M* in;      // Psi at the start
  typename T::M* out;           // Psi after the steps, another buffer
  unsigned int* flag;
};

template <class T>
struct LineTileAcc {
  using C2 = typename T::C;
  const C2* p;   // at the site
  __device__ __forceinline__ C2 at0() const { return p[0]; }
  __device__ __forceinline__ C2 at1(int, int s) const { return p[s]; }
  __device__ __forceinline__ C2 at2(int, int s, int, int t) const { return p[s + t]; }
  __device__ __forceinline__ C2 atv(const int* v) const { return p[v[0]]; }
};

template <class T, int ORDER, int NT, int SPT>
struct Steps1 {
  using R = typename T::R;
  using C = typename T::C;
  using M = typename T::M;
  static constexpr int RW = NT * SPT, W = RW + 4;   // a CTA's sites; with two unused cells at either end

  const Step1Args<T>& A;
  C* buf;              // two stage buffers of W
  int x0;              // grid index of site 0 of the CTA (before any wrap)
  int own_lo, own_hi;  // its own sites, as grid indices
  bool wall_warp;      // this thread is one of the wall warp's
  int site;            // wall warp: the lane's site (-1: none)
  M m[SPT];            // Psi^n
  C K[SPT];
  R v[SPT];            // V at the site F is evaluated at

  __device__ __forceinline__ int wrap(int g) const {
    const int r = g % A.n;
    return r < 0 ? r + A.n : r;
  }

  // The stage's update of the q-th site of the thread, at slot j of the CTA.
  template <int S>
  __device__ __forceinline__ void update(int q, int j, C F, C* out) {
    const C pn = stage_value<T>(m[q]);
    if constexpr (S == 1) K[q] = F;
    if constexpr (S == 2 || S == 3) K[q] = C{fma(R(2), F.x, K[q].x), fma(R(2), F.y, K[q].y)};
    if constexpr (S < 4) {
      out[j + 2] = C{fma(A.dtc[S - 1], F.x, pn.x), fma(A.dtc[S - 1], F.y, pn.y)};
    } else {
      m[q] = final_value<T>(A.dtc[3], K[q], F, m[q]);
      out[j + 2] = stage_value<T>(m[q]);
      const int g = x0 + j;
      if (g >= own_lo && g < own_hi && !(finite_bits(m[q].x) && finite_bits(m[q].y))) atomicOr(A.flag, 1u);
    }
  }

  template <int S, bool WALLS>
  __device__ __forceinline__ void stage(const Field<T>& f, const C* in, C* out) {
    LineTileAcc<T> acc;
    if (WALLS && wall_warp) {
      if (site >= 0) {
        const int g = site, j = g - x0;
        const int c = min(max(g, 1), A.n - 2);   // a boundary site: its interior neighbour
        acc.p = in + j + 2 + (c - g);
        const int idx[1] = {c};
        const C pc = acc.at0();
        const R N = fma(A.s, norm2(pc), -v[0]);
        const C aL = ORDER == 4 ? a_lap_wall<T, 1, ORDER>(f, acc, idx, c, pc, N)
                                : a_lap_body<T, 1, ORDER, LineTileAcc<T>, false>(f, acc, idx, c, pc, N);
        C F = {-fma(N, pc.y, aL.y), fma(N, pc.x, aL.x)};
        if (c != g) {   // see serve_walls
          const C pb = in[j + 2];
          C Fb = {R(0), R(0)};
          if (A.bc == BC_MSD) {
            const R m2 = norm2(pc);
            R theta = R(0);
            if (m2 > A.tiny) theta = fma(F.y, pc.x, -(F.x * pc.y)) / m2;
            Fb = {-theta * pb.y, theta * pb.x};
          } else if (A.bc == BC_L0) {
            const R Nb = fma(A.s, norm2(pb), -ldv<R>(A.V, g));
            Fb = {-Nb * pb.y, Nb * pb.x};
          }
          F = Fb;
        }
        update<S>(0, j, F, out);
      }
    } else if (!wall_warp) {
#pragma unroll
      for (int q = 0; q < SPT; ++q) {
        const int j = threadIdx.x + q * NT, g = x0 + j;
        acc.p = in + j + 2;
        const C pc = acc.at0();
        const R N = fma(A.s, norm2(pc), -v[q]);
        const int idx[1] = {2};
        const C aL = a_lap_body<T, 1, ORDER, LineTileAcc<T>, false>(f, acc, idx, 0, pc, N);
        if (!WALLS || (g >= 2 && g <= A.n - 3))
          update<S>(q, j, C{-fma(N, pc.y, aL.y), fma(N, pc.x, aL.x)}, out);
      }
    }
    __syncthreads();
  }

  template <bool WALLS>
  __device__ __forceinline__ void run(int steps) {
    Field<T> f;
    f.n[0] = A.n;
    f.st[0] = 1;
    f.s = A.s;
    f.h2_over_a = A.h2_over_a;
    f.cL = A.cL;
    f.tiny = A.tiny;
    f.bc = A.bc;
    f.V = A.V;
    C *a = buf, *b = buf + W;
#pragma unroll 1
    for (int i = 0; i < steps; ++i) {
      stage<1, WALLS>(f, a, b);
      stage<2, WALLS>(f, b, a);
      stage<3, WALLS>(f, a, b);
      stage<4, WALLS>(f, b, a);
    }
  }
};

// FP64: the two components of a site on two neighbouring lanes.  GB300 issues one FP64 instruction of a warp
// every 64 cycles per SM sub-partition, however many lanes are active, so a short line's stage takes 64 cycles
// times the FP64 instructions of one thread: 33 for a whole site, 17 for a component (2001 sites, Dirichlet: 6.4 us
// per step with whole sites, 4.8 split).  Lane k of a pair sums the
// stencil of component k and forms t_k = N Psi_k + a Lap Psi_k; since F = i t, it then updates component 1 - k.
template <int ORDER, int SITES>
struct Split1 {
  static constexpr int W = SITES + 4;   // a CTA's sites; with two unused cells at either end

  const Step1Args<P64>& A;
  double* buf;         // two stage buffers of W complex values
  int x0;              // grid index of site 0 of the CTA (before any wrap)
  int own_lo, own_hi;  // its own sites, as grid indices
  bool wall_warp;      // this thread is one of the wall warp's
  int slot;            // the lane pair's site in the CTA (-1: none)
  int k;               // the lane's component
  double m, K, v;      // Psi^n and K_tot of component 1 - k; V at the site F is evaluated at

  __device__ __forceinline__ int wrap(int g) const {
    const int r = g % A.n;
    return r < 0 ? r + A.n : r;
  }

  template <int S, bool WALLS>
  __device__ __forceinline__ void stage(const double* in, double* out) {
    const bool wall = WALLS && wall_warp;
    if (slot >= 0) {   // the same for both lanes of a pair
      const int g = x0 + slot, c = wall ? min(max(g, 1), A.n - 2) : g;
      const double* p = in + 2 * (slot + 2 + (c - g));
      const double pc = p[k], po = p[1 - k], x = k ? po : pc, y = k ? pc : po;
      const double n2 = fma(x, x, y * y), N = fma(A.s, n2, -v);
      double s1 = 0.0;   // a_lap_body, one component
      s1 += (p[2 + k] - pc) + (p[-2 + k] - pc);
      double aL;
      if constexpr (ORDER == 2) {
        aL = A.cL * s1;
      } else {
        double lo, hi;
        auto ghost1 = [&](int dir) {   // ghost() in one dimension
          const double bx = p[2 * dir], by = p[2 * dir + 1], pb = k ? by : bx;
          double fac = 0.0;
          if (A.bc != BC_L0) {
            const double Nb = fma(A.s, fma(bx, bx, by * by), -ldv<double>(A.V, c + dir));
            if (A.bc == BC_DIRICHLET) {
              fac = -A.h2_over_a * Nb;
            } else {
              double ds = 0.0;   // the other component's h^2 D_c
              ds += (p[2 + 1 - k] - po) + (p[-2 + 1 - k] - po);
              const double dx = k ? ds : s1, dy = k ? s1 : ds;
              fac = fma(A.h2_over_a, N - Nb, n2 > A.tiny ? fma(dx, x, dy * y) / n2 : 0.0);
            }
          }
          return fma(2.0, pb, fma(fac, pb, -pc));
        };
        if (!wall || c >= 2) lo = p[-4 + k];
        else lo = ghost1(-1);
        if (!wall || c <= A.n - 3) hi = p[4 + k];
        else hi = ghost1(1);
        double s2 = 0.0;
        s2 += (lo - pc) + (hi - pc);
        aL = A.cL * fma(16.0, s1, -s2);
      }
      double F = fma(N, pc, aL);   // t_k: F_y for k = 0, -F_x for k = 1
      if (wall && c != g) {        // see serve_walls; th: what turns Psi_b into F_b / i
        const double* b = in + 2 * (slot + 2);
        double th = 0.0;
        if (A.bc == BC_MSD) {
          const double o = __shfl_xor_sync(3u << (threadIdx.x & 30), F, 1);   // the pair meets here
          const double Fy = k ? o : F, Fx = -(k ? F : o);
          if (n2 > A.tiny) th = fma(Fy, x, -(Fx * y)) / n2;
        } else if (A.bc == BC_L0) {
          th = fma(A.s, fma(b[0], b[0], b[1] * b[1]), -ldv<double>(A.V, g));
        }
        F = th * b[k];
        if (A.bc == BC_DIRICHLET) F = 0.0;
      }
      if (k) F = -F;
      const int e = 2 * (slot + 2) + 1 - k;
      if (wall || !WALLS || (g >= 2 && g <= A.n - 3)) {
        if constexpr (S == 1) K = F;
        if constexpr (S == 2 || S == 3) K = fma(2.0, F, K);
        if constexpr (S < 4) {
          out[e] = fma(A.dtc[S - 1], F, m);
        } else {
          m = fma(A.dtc[3], K + F, m);
          out[e] = m;
          if (g >= own_lo && g < own_hi && !finite_bits(m)) atomicOr(A.flag, 1u);
        }
      }
    }
    __syncthreads();
  }

  template <bool WALLS>
  __device__ __forceinline__ void run(int steps) {
    double *a = buf, *b = buf + 2 * W;
#pragma unroll 1
    for (int i = 0; i < steps; ++i) {
      stage<1, WALLS>(a, b);
      stage<2, WALLS>(b, a);
      stage<3, WALLS>(a, b);
      stage<4, WALLS>(b, a);
    }
  }
};

}  // namespace nlse
