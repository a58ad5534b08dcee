// 3D stage of the FP32 forms in one launch: columns marching along z with their
// neighbours read through the L1 cache, and the wall sites beside them.
//
// The z-marching tiles of stage_tma.cuh need rows of whole 16 bytes, and their
// walls three more launches on side streams; on grids of a few million sites a
// stage is then as much launches, joins and ring filling as work, and without
// TMA (odd Nx) the cooperative tile loads cost 380 instructions per site.  Here a
// thread owns one column of the deep interior over a chunk of planes: the five
// planes of its own column stay in registers, the eight in-plane neighbours are
// L1 hits (their own columns' threads loaded them two planes ago), all loads
// issued a plane ahead.  What bounds it is the latency of those loads (long
// scoreboard, 48 % issue at four CTAs per SM); 173 instructions per site.  The sites
// next to the walls and the boundary sites are further ranges of blocks, as in
// stage_split.cuh.  The arithmetic is a_lap_body's and rk_apply's on packed FP32
// pairs (stage_step2d.cuh) in the same order: bit-for-bit the other kernels'.
// us per step, MSD 2SHOC, the tiles and this: 203x87x87 FP32 93.7 and 52.6, mixed
// form 112 and 72.3; 100^3 63.9 and 36.9; 128^3 86.6 and 67.5; 160^3 152 and 155;
// 255^3 (no TMA) 667 and 511.
#pragma once
#include "stage_split.cuh"
#include "stage_step2d.cuh"
#include "stage_tma.cuh"

namespace nlse {

constexpr int kMarchTX = 32, kMarchTY = 8;

template <class T, int ORDER, int S>
__global__ void __launch_bounds__(256, 4) k_stage3d_march(const StageArgs<T> A, int ntx, int nty, int zc, unsigned b1,
                                                          unsigned b2, unsigned b3, int64_t n2, int64_t n3, bool walls_first) {
  const Field<T>& f = A.f;
  grid_wait();
  unsigned bi = blockIdx.x;
  if (walls_first) bi = bi < b3 - b1 ? bi + b1 : bi - (b3 - b1);
  if (bi >= b1) {
    if (bi < b2) shell_site<T, 3, ORDER, false, uint32_t>(A, (int64_t)(bi - b1) * 256 + threadIdx.x, n2);
    else boundary_site<T, 3, ORDER, false, uint32_t>(A, (int64_t)(bi - b2) * 256 + threadIdx.x, n3);
    return;
  }
  int b = bi;
  const int tx = b % ntx;
  b /= ntx;
  const int ty = b % nty, tz = b / nty;
  const int gx = 2 + tx * kMarchTX + (int)(threadIdx.x & 31), gy = 2 + ty * kMarchTY + (int)(threadIdx.x >> 5);
  const int zb = 2 + tz * zc, ze = min(zb + zc, f.n[0] - 2);
  if (gx > f.n[2] - 3 || gy > f.n[1] - 3) return;
  const int nx = f.n[2];
  const int64_t plane = (int64_t)f.n[1] * nx;
  int64_t c = zb * plane + (int64_t)gy * nx + gx;
  const float2* in = f.in + c;
  float2 w[5];   // the column's planes z-2 .. z+2 (ordinary loads, see ld2_ordered)
#pragma unroll
  for (int d = 0; d < 4; ++d) w[d] = (ORDER == 4 || d > 0) ? in[(d - 2) * plane] : float2{0.f, 0.f};
  float2 next = in[(ORDER == 4 ? 2 : 1) * plane];
  if (ORDER == 2) { w[3] = next; }
  const bool with_v = f.V != nullptr;
  PointVals<T> pn = load_point<T, S>(A, c, with_v);
  const Pk cL = pk(f.cL), zero = pk(0.f);
  const auto neg = [](float2 v) { return pk(float2{-v.x, -v.y}); };
  // the eight in-plane neighbours, loaded a plane ahead
  float2 xm, xp, ym, yp, xm2, xp2, ym2, yp2;
  auto neighbours = [&]() {
    xm = in[-1];
    xp = in[1];
    ym = in[-nx];
    yp = in[nx];
    if constexpr (ORDER == 4) {
      xm2 = in[-2];
      xp2 = in[2];
      ym2 = in[-2 * nx];
      yp2 = in[2 * nx];
    }
  };
  neighbours();
  for (int z = zb; z < ze; ++z) {
    const PointVals<T> p = pn;
    if (ORDER == 4) w[4] = next;
    else w[3] = next;
    if (z + 1 < ze) {
      next = in[(ORDER == 4 ? 3 : 2) * plane];
      pn = load_point<T, S>(A, c + plane, with_v);
    }
    const float2 pc = w[2];
    const Pk m = neg(pc);
    Pk s1 = add(add(pk(w[3]), m), add(pk(w[1]), m));   // z, y, x as a_lap_body
    s1 = add(s1, zero);                                // its first sum starts from +0
    s1 = add(s1, add(add(pk(yp), m), add(pk(ym), m)));
    s1 = add(s1, add(add(pk(xp), m), add(pk(xm), m)));
    Pk aL;
    if constexpr (ORDER == 2) {
      aL = mul(cL, s1);
    } else {   // -s2: the differences the other way round
      const Pk q = pk(pc);
      Pk s2 = add(add(q, neg(w[0])), add(q, neg(w[4])));
      s2 = add(s2, add(add(q, neg(ym2)), add(q, neg(yp2))));
      s2 = add(s2, add(add(q, neg(xm2)), add(q, neg(xp2))));
      aL = mul(cL, fma_(pk(16.f), s1, s2));
    }
    in += plane;
    if (z + 1 < ze) neighbours();
    const float N = fma(f.s, norm2(pc), -p.v);
    const float2 t = unpk(fma_(pk(N), pk(pc), aL));   // F = i t
    rk_apply<T, S>(A, c, {-t.y, t.x}, p);
#pragma unroll
    for (int d = 0; d < 4; ++d) w[d] = w[d + 1];
    c += plane;
  }
}

template <class T, int ORDER, int S>
cudaError_t launch_march_stage(const StageArgs<T>& A, cudaStream_t stream) {
  auto kern = k_stage3d_march<T, ORDER, S>;
  static const int per_sm = resident_per_sm(kern, 256, 0);
  const int ntx = (A.f.n[2] - 4 + kMarchTX - 1) / kMarchTX, nty = (A.f.n[1] - 4 + kMarchTY - 1) / kMarchTY;
  const int planes = A.f.n[0] - 4;
  // The wall blocks first and the columns in two waves behind them, or the columns in one wave and the wall blocks
  // after it: the second for the mixed form above 2^20 sites (us per step, two waves and one, MSD 2SHOC: 100^3 48.8 and
  // 50.5, 104^3 63.3 and 63.6, 110^3 68.4 and 66.0, 203x87x87 75.9 and 73.2, 140x120x130 95.9 and 88.7, 143^3 141 and
  // 132; against it 128^3 96.7 and 103.5, 300x64x64 71.0 and 78.0).  FP32: 128^3 72.6 and 81.4, 143^3 104.6 and 94.8.
  const bool one_wave = !std::is_same<typename T::M, typename T::C>::value && A.f.ninterior > (int64_t(1) << 20);
  int nzc = z_chunks(ntx * nty, planes, one_wave ? per_sm : 2 * per_sm, 3);
  const int zc = (planes + nzc - 1) / nzc;
  nzc = (planes + zc - 1) / zc;
  const int64_t deep = (int64_t)planes * (A.f.n[1] - 4) * (A.f.n[2] - 4);
  const int64_t n2 = A.f.ninterior - deep, n3 = boundary_count(3, A.f.n, A.f.m);
  const unsigned b1 = (unsigned)(ntx * nty * nzc), b2 = b1 + (unsigned)((n2 + 255) / 256), b3 = b2 + (unsigned)((n3 + 255) / 256);
  return launch_early(true, kern, dim3(b3), dim3(256), 0, stream, A, ntx, nty, zc, b1, b2, b3, n2, n3, !one_wave);
}

// Walls on every side and a deep interior (every extent >= 5); fewer than 2^31 sites.
inline bool march_ok(const int* n, int bc) {
  return bc != BC_PERIODIC && n[0] >= 5 && n[1] >= 5 && n[2] >= 5 && (int64_t)n[0] * n[1] * n[2] < (int64_t(1) << 31);
}

// Flat grids that are mostly MSD walls: with a thread per boundary site (walls_apart) they are slower than the tiles
// with a thread per wall site (2SHOC, this form and that: 6x600x700 142 and 131, 700x6x700 198 and 173; 6x300x300 38
// and 43, 700x700x6 410 and 470; central differences with V 6x500x1000 126 and 119, without 6x600x700 86 and 97).
template <int ORDER, class T>
inline bool march_thin(const Field<T>& f) {
  return f.bc == BC_MSD && (f.n[0] < 8 || f.n[1] < 8) && boundary_count(3, f.n, f.m) > (ORDER == 4 ? 500000 : 900000);
}

// Whether the steps of a grid take the columns: a few million sites, or rows that TMA cannot take (the figures above).
template <int ORDER, class T>
inline bool march_serves(const Field<T>& f, bool tma) {
  const bool small = (int64_t)f.n[0] * f.n[1] * f.n[2] <= 3000000 && !march_thin<ORDER>(f);
  return (small || !tma) && march_ok(f.n, f.bc);
}

template <class T, int ORDER>
cudaError_t launch_march(const StageArgs<T>& A, cudaStream_t stream) {
  switch (A.stage) {
    case 1: return launch_march_stage<T, ORDER, 1>(A, stream);
    case 2: return launch_march_stage<T, ORDER, 2>(A, stream);
    case 3: return launch_march_stage<T, ORDER, 3>(A, stream);
    default: return launch_march_stage<T, ORDER, 4>(A, stream);
  }
}

}  // namespace nlse
