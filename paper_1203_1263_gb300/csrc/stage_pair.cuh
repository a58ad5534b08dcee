// The per-site FP64 stage of a small 3D grid with the two components of a site
// on neighbouring lanes.
//
// GB300 issues one FP64 instruction of a warp every 64 cycles per SM
// sub-partition, however many lanes are active, so on a grid that fills the
// sub-partitions with about one warp each a stage takes 64 cycles times the FP64
// instructions of a thread's chain.  A lane here carries the stencil of component
// k (half the chain) and forms t_k = N Psi_k + a Lap Psi_k; since F = i t, it then
// updates component 1 - k.  The deep sites, the sites next to a wall and the
// boundary sites are three ranges of blocks as in stage_split.cuh.  Beyond that
// the chain is shortened where the lanes meet a wall: an axis has one ghost
// whichever of its two walls it is (both only when one interior cell separates
// them), its operands are requested with the site's own, and the MSD ratio
// (D_c / Psi_c) is divided out once per site.  The sums and products are
// site_rhs's, ghost's and rk_apply's in the same order: bit-for-bit the other
// kernels' results.  A CTA of four warps puts one on each sub-partition.  There is
// no launch_dependents: CTAs of the next stage that arrive while this one's still
// run are placed two to an SM on the SMs that finish first, and two of the
// long chains on one sub-partition take twice the time (21^3: 50.7 us per step).
// What bounds it at 21^3 is the chain of the boundary sites and four launches.
// us per step, MSD walls, one thread per site and this: 2SHOC 16^3 34.5 and 21.6,
// 21^3 37.7 and 21.8, 32^3 44.0 and 38.8, 46^3 101.8 and 74.5, 80^3 314 and 298,
// 100^3 529 and 556; central differences 16^3 13.5 and 12.1, 21^3 14.4 and 12.5,
// 26^3 14.1 and 14.4, 32^3 17.8 and 19.8 (more sites only pay the terms that both
// lanes compute).
#pragma once
#include "stage_split.cuh"

namespace nlse {

// t_k at interior site c; WALL: c may be next to a wall.  *pc: Psi_c; *m2: |Psi_c|^2.
// Every lane of the warp calls it with its partner's c.
template <int ORDER, bool WALL>
__device__ __forceinline__ double pair_rhs(const Field<P64>& f, const int* idx, int64_t c, int k, double2* pc_out, double* m2_out) {
  constexpr int D = 3;
  const double* in = reinterpret_cast<const double*>(f.in) + k;   // component k of the field
  auto at = [&](int64_t i) { return in[2 * i]; };   // ordinary loads, see ld2_ordered
  const double2 pc = f.in[c];
  const double v = ldv<double>(f.V, c);
  double u1[D], w1[D], hi[D], lo[D];
  double2 pb[D];
  double vb[D], gu[D][D], gw[D][D];
  bool wlo[D], whi[D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    u1[a] = at(c + f.st[a]);
    w1[a] = at(c - f.st[a]);
    wlo[a] = WALL && idx[a] == 1;
    whi[a] = WALL && idx[a] == f.n[a] - 2;
    if constexpr (ORDER == 4) {
      hi[a] = at(c + (whi[a] ? 1 : 2) * f.st[a]);
      lo[a] = at(c - (wlo[a] ? 1 : 2) * f.st[a]);
    }
  }
  // a wall's ghost operands, of the lower wall first
  auto load_wall = [&](int a, int64_t d) {
    const int64_t b = c + d;
    pb[a] = f.in[b];
    vb[a] = ldv<double>(f.V, b);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      if (j == a) continue;
      gu[a][j] = at(b + f.st[j]);
      gw[a][j] = at(b - f.st[j]);
    }
  };
  if constexpr (WALL && ORDER == 4) {
#pragma unroll
    for (int a = 0; a < D; ++a)
      if (wlo[a] || whi[a]) load_wall(a, wlo[a] ? -f.st[a] : f.st[a]);
  }
  const double pk = k ? pc.y : pc.x;
  const double m2 = norm2(pc), N = fma(f.s, m2, -v);
  *pc_out = pc;
  *m2_out = m2;
  double s1 = 0.0;   // see a_lap_body
#pragma unroll
  for (int a = 0; a < D; ++a) s1 += (u1[a] - pk) + (w1[a] - pk);
  if constexpr (ORDER == 2) {
    return fma(N, pk, f.cL * s1);
  } else {
    if constexpr (WALL) {
      double ratio = 0.0;
      if (f.bc == BC_MSD) {
        const double o = __shfl_xor_sync(0xffffffffu, s1, 1);
        const double dx = k ? o : s1, dy = k ? s1 : o;
        if (m2 > f.tiny) ratio = fma(dx, pc.x, dy * pc.y) / m2;
      }
      auto ghost1 = [&](int a) {   // see ghost
        double fac = 0.0;
        if (f.bc != BC_L0) {
          const double Nb = fma(f.s, norm2(pb[a]), -vb[a]);
          fac = f.bc == BC_DIRICHLET ? -f.h2_over_a * Nb : fma(f.h2_over_a, N - Nb, ratio);
        }
        const double b = k ? pb[a].y : pb[a].x;
        double g = fma(2.0 * D, b, fma(fac, b, -pk));
#pragma unroll
        for (int j = 0; j < D; ++j)
          if (j != a) g -= gu[a][j] + gw[a][j];
        return g;
      };
#pragma unroll
      for (int a = 0; a < D; ++a) {
        if (wlo[a] || whi[a]) {
          const double g = ghost1(a);
          if (wlo[a]) lo[a] = g;
          else hi[a] = g;
        }
        if (wlo[a] && whi[a]) {
          load_wall(a, f.st[a]);
          hi[a] = ghost1(a);
        }
      }
    }
    double s2 = 0.0;
#pragma unroll
    for (int a = 0; a < D; ++a) s2 += (lo[a] - pk) + (hi[a] - pk);
    return fma(N, pk, f.cL * fma(16.0, s1, -s2));
  }
}

// rk_apply for the j-th value of the fields seen as reals.
__device__ __forceinline__ unsigned int pair_apply(const StageArgs<P64>& A, int64_t j, double F) {
  auto r = [](const double2* p) { return reinterpret_cast<const double*>(p); };
  auto w = [](double2* p) { return reinterpret_cast<double*>(p); };
  switch (A.stage) {
    case 0: w(A.out)[j] = A.dtc * F; break;
    case 1:
      w(A.ktot)[j] = F;
      w(A.out)[j] = fma(A.dtc, F, r(A.psin)[j]);
      break;
    case 2:
    case 3:
      w(A.ktot)[j] = fma(2.0, F, w(A.ktot)[j]);
      w(A.out)[j] = fma(A.dtc, F, r(A.psin)[j]);
      break;
    default: {
      const double q = fma(A.dtc, w(A.ktot)[j] + F, r(A.master_in)[j]);
      w(A.master)[j] = q;
      if (!finite_bits(q)) atomicOr(A.flag, 1u);
      return range_bits(q);
    }
  }
  return 0u;
}

// Blocks [0, b1): the n3 boundary sites, whose chain is the longest; [b1, b2): the n2 sites next to a wall; the rest:
// the n1 deep sites.  Lanes past the end repeat the range's last site and store nothing.
template <int ORDER>
__global__ void __launch_bounds__(128) k_stage_pair(const StageArgs<P64> A, unsigned b1, unsigned b2, int n1, int n2, int n3) {
  const Field<P64>& f = A.f;
  const int kind = blockIdx.x < b1 ? 0 : (blockIdx.x < b2 ? 1 : 2), n = kind == 0 ? n3 : (kind == 1 ? n2 : n1);
  const int t0 = (int)(blockIdx.x - (kind == 0 ? 0 : (kind == 1 ? b1 : b2))) * (int)(blockDim.x >> 1) + (int)(threadIdx.x >> 1);
  const int k = threadIdx.x & 1;
  const uint32_t t = min(t0, n - 1);
  int idx[3];
  int64_t site, c;   // the site to update; the interior site F is evaluated at
  if (kind == 0) {
    site = boundary_decode<P64, 3, uint32_t>(f, t, idx);
    c = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      idx[a] = min(max(idx[a], 1), f.n[a] - 2);
      c += idx[a] * f.st[a];
    }
  } else if (kind == 1) {
    site = c = shell_decode<P64, 3, uint32_t>(f, t, idx);
  } else {
    uint32_t rem = t;
    c = 0;
#pragma unroll
    for (int a = 2; a >= 0; --a) {
      const uint32_t m = f.n[a] - 4, q = rem / m;
      idx[a] = int(rem - q * m) + 2;
      rem = q;
      c += idx[a] * f.st[a];
    }
    site = c;
  }
  grid_wait();
  double F = 0.0;   // t_k first: F_y for k = 0, -F_x for k = 1
  double2 pc;
  double m2;
  if (kind == 2) {
    F = pair_rhs<ORDER, false>(f, idx, c, k, &pc, &m2);
  } else if (kind == 1 || f.bc == BC_MSD) {
    F = pair_rhs<ORDER, true>(f, idx, c, k, &pc, &m2);
  }
  if (kind == 0 && f.bc != BC_DIRICHLET) {   // see serve_walls
    const double2 pb = f.in[site];
    double th = 0.0;                         // what turns Psi_b into F_b / i
    if (f.bc == BC_MSD) {
      const double o = __shfl_xor_sync(0xffffffffu, F, 1);
      const double Fy = k ? o : F, Fx = -(k ? F : o);
      if (m2 > f.tiny) th = fma(Fy, pc.x, -(Fx * pc.y)) / m2;
    } else {
      th = fma(f.s, norm2(pb), -ldv<double>(f.V, site));
    }
    F = th * (k ? pb.y : pb.x);
  }
  if (k && !(kind == 0 && f.bc == BC_DIRICHLET)) F = -F;
  unsigned int ex = 0;
  if (t0 < n) ex = pair_apply(A, 2 * site + 1 - k, F);
  if (A.emax) emax_commit(A.emax, ex);
}

template <int ORDER>
cudaError_t launch_pair(const StageArgs<P64>& A, cudaStream_t stream) {
  int n1 = 1;
  for (int k = 0; k < 3; ++k) n1 *= A.f.n[k] > 4 ? A.f.n[k] - 4 : 0;
  const int n2 = (int)A.f.ninterior - n1, n3 = (int)boundary_count(3, A.f.n, A.f.m);
  constexpr int threads = 128, per = threads / 2;
  const unsigned b1 = (n3 + per - 1) / per, b2 = b1 + (n2 + per - 1) / per, b3 = b2 + (n1 + per - 1) / per;
  return launch_early(true, k_stage_pair<ORDER>, dim3(b3), dim3(threads), 0, stream, A, b1, b2, n1, n2, n3);
}

}  // namespace nlse
