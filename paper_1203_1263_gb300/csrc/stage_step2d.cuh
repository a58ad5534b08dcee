// A whole RK4 step of a 2D grid in one pass over memory.
//
// Streaming the four stages of Eq. RK4_GPU through memory moves K_tot,
// Psi_tmp and Psi_out in and out three times each (152 bytes per site and step
// in FP32 with V) and takes eight launches.  Here a CTA takes a TX x TY tile
// through all four stages: it loads Psi^n (and V) of the tile plus an
// eight-cell halo once, evaluates stage 1 on the tile plus six cells, stage 2
// on the tile plus four, stage 3 plus two and stage 4 on the tile alone, each
// from the one before in shared memory, and writes Psi^{n+1}.  What bounds it
// is the shared-memory and issue rate of the stages (the halo costs a factor
// 1.3-1.7 in evaluated sites; on a batch of uneven grids the shared-memory pipe
// is 72 % busy and the issue slots 46 %, the rest is barriers at the end of a
// stage), not memory: 20 bytes per site and step.  Measured, us per step, four
// launches per stage pass before and now: 1000^2 FP32, central differences,
// MSD, 30.6 and 15.8; on small grids the launches and the four stages' latency
// remain (100^2: 6.9).
// Psi^{n+1} goes to another buffer than Psi^n, because neighbouring tiles
// still read Psi^n.
//
// Sites are computed two at a time (pairs along x, 16-byte shared-memory
// accesses) in strips of RY rows with no wall logic at all: where the five-point
// 2SHOC form reaches past a wall, the cell beyond it in the tile first gets the
// ghost value that serves there (ghost() of nlse_device.cuh), one thread per wall
// site, and the boundary cells, which the strips fill with values of no meaning,
// are set afterwards, one thread per boundary site.  A tile away from the walls
// skips both.  (Wall sites as a branch of the site code, as the per-site kernel
// has it, doubled a small grid's step: 9.9 against 6.2 us for the same grid
// without walls at 256^2.)  Every site's arithmetic is the per-site kernels' in
// the same order, so results are bit-for-bit theirs.
#pragma once
#include "nlse_device.cuh"

namespace nlse {

constexpr int kStepHalo = 8;   // two cells per stage

// Everything one step needs (T: P32 or PMix).
template <class T>
struct Step2Args {
  using R = typename T::R;
  int n[2];                     // (Ny, Nx)
  int bc;
  R s, h2_over_a, cL, tiny;     // as in Field
  R dtc[4];                     // dt/2, dt/2, dt, dt/6
  const typename T::VR* V;      // or nullptr
  const typename T::M* in;      // Psi^n
  typename T::M* out;           // Psi^{n+1}, another buffer
  unsigned int* flag;
};

// Shared memory of a TX x ty tile with its halo: Psi^n and the two stage buffers, K_tot on the tile and on the
// boundary sites along its walls, V if there is one.
template <int TX>
inline size_t step2_smem(int ty, bool with_v) {
  const size_t W = TX + 2 * kStepHalo, ps = W * (ty + 2 * kStepHalo);
  return (3 * ps + W * ty + 2 * (W + ty + 2 * kStepHalo)) * sizeof(float2) + (with_v ? ps * sizeof(float) : 0);
}

// A complex FP32 value as one packed operand: sm_100's add, mul and fma on two FP32 lanes round each lane
// like the scalar instruction, so the deep sites' arithmetic below is a_lap_body's and rk_apply's bit for
// bit at half the instructions.
struct Pk { unsigned long long v; };
__device__ __forceinline__ Pk pk(float2 a) {
  Pk r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a.x), "f"(a.y));
  return r;
}
__device__ __forceinline__ Pk pk(float a) { return pk(float2{a, a}); }
__device__ __forceinline__ float2 unpk(Pk a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ Pk add(Pk a, Pk b) {
  Pk r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ Pk mul(Pk a, Pk b) {
  Pk r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ Pk fma_(Pk a, Pk b, Pk c) {
  Pk r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// Single sites (wall code): operands straight from the tile.
template <class LT, int W>
struct TileAcc2 {
  using C2 = typename LT::C;
  const C2* p;
  int o;
  __device__ __forceinline__ static int off(int k, int s) { return k == 0 ? s * W : s; }
  __device__ __forceinline__ C2 at0() const { return p[o]; }
  __device__ __forceinline__ C2 at1(int k, int s) const { return p[o + off(k, s)]; }
  __device__ __forceinline__ C2 at2(int k, int s, int j, int t) const { return p[o + off(k, s) + off(j, t)]; }
  __device__ __forceinline__ C2 atv(const int* v) const { return p[o + v[0] * W + v[1]]; }
};

// Two neighbouring complex values, 16 bytes at a time.
struct Pair2 { float2 a, b; };
__device__ __forceinline__ Pair2 ld_pair(const float2* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ void st_pair(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_pair(double2* p, double2 a, double2 b) {
  p[0] = a;
  p[1] = b;
}

// Psi^n in stage precision, and Psi^{n+1} in the master's.
template <class T>
__device__ __forceinline__ typename T::C stage_value(const typename T::M m) {
  if constexpr (std::is_same<typename T::M, typename T::C>::value) return m;
  else return typename T::C{d2f_rn(m.x), d2f_rn(m.y)};
}
template <class T>
__device__ __forceinline__ typename T::M final_value(typename T::R dtc, typename T::C K, typename T::C F,
                                                     typename T::M pn) {
  typename T::M q;   // as rk_apply's stage 4
  if constexpr (std::is_same<typename T::M, typename T::C>::value) {
    q.x = fma(dtc, K.x + F.x, pn.x);
    q.y = fma(dtc, K.y + F.y, pn.y);
  } else {
    const float ix = dtc * (K.x + F.x), iy = dtc * (K.y + F.y);
    q.x = pn.x + f2d_exact(ix);
    q.y = pn.y + f2d_exact(iy);
  }
  return q;
}

// ty (the tile's rows) is a multiple of RY.  WRAP: the grid is periodic.
template <class T, int ORDER, int TX, int NT, int RY, bool WRAP>
struct Step2Tile {
  using LT = L32;
  using C = float2;
  using R = float;
  using M = typename T::M;
  static constexpr int HALO = kStepHalo, W = TX + 2 * HALO;
  static constexpr bool kMaster = !std::is_same<M, C>::value;   // an FP64 master over FP32 stages

  const Step2Args<T>& A;
  C *P, *a, *b, *K;      // Psi^n; the two stage buffers; K_tot
  C *Krow, *Kcol;        // K_tot at the boundary sites on the low and high y walls, x walls
  R* V;
  const int TY;          // rows of the tile
  const int PS;          // elements of the tile with its halo
  int ox, oy;            // grid coordinates of the tile's element (0, 0)
  bool with_v;

  __device__ __forceinline__ Step2Tile(const Step2Args<T>& A_, int rows, int tx, int ty, unsigned char* smem)
      : A(A_), TY(rows), PS(W * (rows + 2 * HALO)) {
    P = reinterpret_cast<C*>(smem);
    a = P + PS;
    b = a + PS;
    K = b + PS;
    Krow = K + W * TY;
    Kcol = Krow + 2 * W;
    V = reinterpret_cast<R*>(Kcol + 2 * (TY + 2 * HALO));
    ox = tx * TX - HALO;
    oy = ty * TY - HALO;
    with_v = A.V != nullptr;
  }

  // Copy a tile's rows from global memory (elements of B bytes; zero outside the grid, wrapped on a periodic
  // one), a warp per row, without going through registers; wait with arrive().
  template <int B>
  __device__ __forceinline__ void copy_rows(void* dst, const void* src) const {
    const int ny = A.n[0], nx = A.n[1], H = TY + 2 * HALO;
    const int lane = threadIdx.x & 31;
    const uint32_t d0 = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    const char* s0 = static_cast<const char*>(src);
    const bool wrap_x = WRAP && (ox < 0 || ox + W > nx);
    const int x0 = wrap_x ? ((ox % nx) + nx) % nx : ox;   // column of the tile's first one
    for (int r = threadIdx.x >> 5; r < H; r += NT / 32) {
      int gy = oy + r;
      if (WRAP && (gy < 0 || gy >= ny)) gy = ((gy % ny) + ny) % ny;
      const bool in_y = gy >= 0 && gy < ny;
      const char* row = s0 + ((int64_t)(in_y ? gy : 0) * nx) * B;
      if (wrap_x) {   // only the tiles at an end of the rows (1000^2 FP32: 37 us per step with every column wrapped)
        for (int q = lane; q < W; q += 32) {
          const int g = x0 + q, gx = nx >= W ? (g >= nx ? g - nx : g) : g % nx;
          copy_async<B>(d0 + (r * W + q) * B, row + (int64_t)gx * B, B);
        }
        continue;
      }
#pragma unroll
      for (int q0 = 0; q0 < W; q0 += 32) {
        const int q = q0 + lane, gx = ox + q;
        const bool ok = in_y && gx >= 0 && gx < nx;
        if (q < W) copy_async<B>(d0 + (r * W + q) * B, row + (ok ? (int64_t)gx * B : 0), ok ? B : 0);
      }
    }
  }
  // cp.async of B bytes, n of them read and the rest zero.
  template <int B>
  __device__ __forceinline__ static void copy_async(uint32_t dst, const void* src, int n) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(B), "r"(n) : "memory");
  }
  __device__ __forceinline__ static void arrive() {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }

  __device__ __forceinline__ void load_potential() {
    if (with_v) copy_rows<sizeof(float)>(V, A.V);
  }
  __device__ __forceinline__ void load() {
    // an FP64 master goes through the two stage buffers (one after the other) and is rounded from there
    copy_rows<sizeof(M)>(kMaster ? a : P, A.in);
    arrive();
    if constexpr (kMaster) {
      const M* m = reinterpret_cast<const M*>(a);
      for (int e = threadIdx.x; e < PS; e += NT) P[e] = stage_value<T>(m[e]);
      __syncthreads();
    }
  }

  // The update of boundary site e (grid index g), its K_tot at k.
  template <int S>
  __device__ __forceinline__ void update_boundary(C* out, int e, int64_t g, C* k, bool own, C F) {
    if constexpr (S < 4) {
      if (S == 1) *k = F;
      else *k = C{fma(R(2), F.x, k->x), fma(R(2), F.y, k->y)};
      const C pn = P[e];
      out[e] = C{fma(A.dtc[S - 1], F.x, pn.x), fma(A.dtc[S - 1], F.y, pn.y)};
    } else if (own) {
      M pn;
      if constexpr (kMaster) pn = A.in[g];
      else pn = P[e];
      const M q = final_value<T>(A.dtc[3], *k, F, pn);
      A.out[g] = q;
      if (!(finite_bits(q.x) && finite_bits(q.y))) atomicOr(A.flag, 1u);
    }
  }

  // a Lap Psi at a deep site from its neighbours (a_lap_body's order: y before x).
  struct Nbr { C ym2, ym, yp, yp2, xm2, xm, xp, xp2; };
  __device__ __forceinline__ Pk lap(C c, const Nbr& n) const {
    const Pk m = pk(C{-c.x, -c.y});
    Pk s1 = add(add(pk(n.yp), m), add(pk(n.ym), m));
    s1 = add(s1, pk(0.f));   // the scalar code's first sum starts from +0
    s1 = add(s1, add(add(pk(n.xp), m), add(pk(n.xm), m)));
    const Pk cL = pk(A.cL);
    if constexpr (ORDER == 2) return mul(cL, s1);
    const Pk p = pk(c);      // -s2: the differences the other way round
    const auto neg = [](C v) { return pk(C{-v.x, -v.y}); };
    Pk s2 = add(add(p, neg(n.ym2)), add(p, neg(n.yp2)));
    s2 = add(s2, add(add(p, neg(n.xm2)), add(p, neg(n.xp2))));
    return mul(cL, fma_(pk(16.f), s1, s2));
  }

  // One deep site's stage: t = N Psi + a Lap Psi (so F = i t), K_tot in units of t.
  __device__ __forceinline__ C rhs(C c, const Nbr& n, R v) const {
    const R N = fma(A.s, norm2(c), -v);
    return unpk(fma_(pk(N), pk(c), lap(c, n)));
  }

  // RY rows of two sites each, starting at element e (grid index g and coordinates: stage 4 only).
  template <int S, bool WALLS>
  __device__ __forceinline__ void strip(const C* in, C* out, int e, int64_t g, int gy, int gx, bool own_x, int ly, bool vec) {
    Pair2 col[RY + 4];
#pragma unroll
    for (int r = ORDER == 4 ? 0 : 1; r < (ORDER == 4 ? RY + 4 : RY + 3); ++r) col[r] = ld_pair(in + e + (r - 2) * W);
    const int lo = WRAP ? 0 : 1;   // first updated index
    const bool m0 = !WALLS || (gx >= lo && gx < A.n[1] - lo), m1 = !WALLS || (gx + 1 >= lo && gx + 1 < A.n[1] - lo);
#pragma unroll
    for (int r = 0; r < RY; ++r) {
      const int er = e + r * W;
      const Pair2 c = col[r + 2];
      const Pair2 l = ld_pair(in + er - 2), q = ld_pair(in + er + 2);
      R v0 = R(0), v1 = R(0);
      if (with_v) {
        const float2 v = *reinterpret_cast<const float2*>(V + er);
        v0 = v.x;
        v1 = v.y;
      }
      const C t0 = rhs(c.a, Nbr{col[r].a, col[r + 1].a, col[r + 3].a, col[r + 4].a, l.a, l.b, c.b, q.a}, v0);
      const C t1 = rhs(c.b, Nbr{col[r].b, col[r + 1].b, col[r + 3].b, col[r + 4].b, l.b, c.a, q.a, q.b}, v1);
      const C F0 = {-t0.y, t0.x}, F1 = {-t1.y, t1.x};
      if constexpr (S < 4) {
        if (own_x && unsigned(ly + r - HALO) < unsigned(TY)) {
          C* k = K + (er - HALO * W);
          if (S == 1) {
            st_pair(k, F0, F1);
          } else {
            const Pair2 o = ld_pair(k);
            st_pair(k, unpk(fma_(pk(2.f), pk(F0), pk(o.a))), unpk(fma_(pk(2.f), pk(F1), pk(o.b))));
          }
        }
        const Pair2 pn = ld_pair(P + er);
        const Pk h = pk(A.dtc[S - 1]);
        st_pair(out + er, unpk(fma_(h, pk(F0), pk(pn.a))), unpk(fma_(h, pk(F1), pk(pn.b))));
      } else {
        const int64_t gr = g + (int64_t)r * A.n[1];
        const bool my = !WALLS || (gy + r >= lo && gy + r < A.n[0] - lo);
        const Pair2 k = ld_pair(K + (er - HALO * W));
        M p0, p1;
        if constexpr (kMaster) {
          p0 = p1 = M{0, 0};
          if (my && m0) p0 = A.in[gr];
          if (my && m1) p1 = A.in[gr + 1];
        } else {
          const Pair2 pn = ld_pair(P + er);
          p0 = pn.a;
          p1 = pn.b;
        }
        const M q0 = final_value<T>(A.dtc[3], k.a, F0, p0), q1 = final_value<T>(A.dtc[3], k.b, F1, p1);
        if (my && m0 && m1 && vec) {
          st_pair(A.out + gr, q0, q1);
        } else {
          if (my && m0) A.out[gr] = q0;
          if (my && m1) A.out[gr + 1] = q1;
        }
        bool bad = my && m0 && !(finite_bits(q0.x) && finite_bits(q0.y));
        bad |= my && m1 && !(finite_bits(q1.x) && finite_bits(q1.y));
        if (bad) atomicOr(A.flag, 1u);
      }
    }
  }

  __device__ __forceinline__ Field<LT> wall_field() const {
    Field<LT> f;
    f.n[0] = A.n[0]; f.n[1] = A.n[1];
    f.st[0] = W; f.st[1] = 1;
    f.s = A.s;
    f.h2_over_a = A.h2_over_a;
    f.cL = A.cL;
    f.tiny = A.tiny;
    f.bc = A.bc;
    f.V = with_v ? reinterpret_cast<const OnChip<R>*>(V) : nullptr;
    return f;
  }

  // The interior sites of the stage's region, clipped to the grid, and which walls they touch.
  struct Clip { int ylo, yhi, xlo, xhi; bool top, bot, left, right; };
  template <int S>
  __device__ __forceinline__ Clip clip() const {
    constexpr int e0 = 2 * (4 - S);
    Clip c;
    c.ylo = max(oy + HALO - e0, 1);
    c.yhi = min(oy + HALO + TY + e0, A.n[0] - 1);
    c.xlo = max(ox + HALO - e0, 1);
    c.xhi = min(ox + HALO + TX + e0, A.n[1] - 1);
    c.top = c.ylo == 1;
    c.bot = c.yhi == A.n[0] - 1;
    c.left = c.xlo == 1;
    c.right = c.xhi == A.n[1] - 1;
    return c;
  }

  // The ghosts of the stage input beyond the walls, into the cells two beyond the sites next to them.
  template <int S>
  __device__ __forceinline__ void ghosts(C* in) {
    const Clip c = clip<S>();
    const Field<LT> f = wall_field();
    const int rw = c.xhi - c.xlo, rh = c.yhi - c.ylo;
    const int n0 = c.top ? rw : 0, n1 = n0 + (c.bot ? rw : 0), n2 = n1 + (c.left ? rh : 0), n3 = n2 + (c.right ? rh : 0);
#pragma unroll 1
    for (int t = threadIdx.x; t < n3; t += NT) {
      const bool row = t < n1, hi = row ? t >= n0 : t >= n2;
      const int gy = row ? (hi ? A.n[0] - 2 : 1) : c.ylo + (t - (hi ? n2 : n1));
      const int gx = row ? c.xlo + (t - (hi ? n0 : 0)) : (hi ? A.n[1] - 2 : 1);
      const int e = (gy - oy) * W + (gx - ox);
      TileAcc2<LT, W> acc;
      acc.p = in;
      acc.o = e;
      const C pc = in[e], u = in[e + W], w = in[e - W], q = in[e + 1], l = in[e - 1];
      const R Nc = fma(A.s, norm2(pc), -(with_v ? V[e] : R(0)));
      C dh = {R(0), R(0)};   // h^2 D_c as a_lap_body sums it
      dh.x += (u.x - pc.x) + (w.x - pc.x);
      dh.y += (u.y - pc.y) + (w.y - pc.y);
      dh.x += (q.x - pc.x) + (l.x - pc.x);
      dh.y += (q.y - pc.y) + (l.y - pc.y);
      const int dir = hi ? 1 : -1;
      C g;
      if (row) g = ghost<LT, 2>(f, acc, 0, dir, e, pc, dh, Nc);
      else g = ghost<LT, 2>(f, acc, 1, dir, e, pc, dh, Nc);
      in[e + 2 * dir * (row ? W : 1)] = g;
    }
  }

  // The boundary sites next to the stage's region, each with its nearest interior site's F (see serve_walls).
  template <int S>
  __device__ __forceinline__ void boundary(const C* in, C* out) {
    const Clip c = clip<S>();
    const int x0 = c.xlo - (c.left ? 1 : 0), x1 = c.xhi + (c.right ? 1 : 0);   // rows with their corners
    const int rw = x1 - x0, rh = c.yhi - c.ylo;
    const int n0 = c.top ? rw : 0, n1 = n0 + (c.bot ? rw : 0), n2 = n1 + (c.left ? rh : 0), n3 = n2 + (c.right ? rh : 0);
#pragma unroll 1
    for (int t = threadIdx.x; t < n3; t += NT) {
      const bool row = t < n1, hi = row ? t >= n0 : t >= n2;
      const int by = row ? (hi ? A.n[0] - 1 : 0) : c.ylo + (t - (hi ? n2 : n1));
      const int bx = row ? x0 + (t - (hi ? n0 : 0)) : (hi ? A.n[1] - 1 : 0);
      const int cy = min(max(by, 1), A.n[0] - 2), cx = min(max(bx, 1), A.n[1] - 2);
      const int eb = (by - oy) * W + (bx - ox);
      C Fb = {R(0), R(0)};
      if (A.bc == BC_MSD) {   // F at the interior site once more, from its own operands
        const int e = (cy - oy) * W + (cx - ox);
        const C pc = in[e], pb = in[eb];
        Nbr n;
        n.ym = in[e - W]; n.yp = in[e + W];
        n.xm = in[e - 1]; n.xp = in[e + 1];
        if constexpr (ORDER == 4) {
          n.ym2 = in[e - 2 * W]; n.yp2 = in[e + 2 * W];
          n.xm2 = in[e - 2]; n.xp2 = in[e + 2];
        }
        const C tt = rhs(pc, n, with_v ? V[e] : R(0)), F = {-tt.y, tt.x};
        const R m2 = norm2(pc);
        R theta = R(0);
        if (m2 > A.tiny) theta = fma(F.y, pc.x, -(F.x * pc.y)) / m2;
        Fb = {-theta * pb.y, theta * pb.x};
      } else if (A.bc == BC_L0) {
        const C pb = in[eb];
        const R Nb = fma(A.s, norm2(pb), -(with_v ? V[eb] : R(0)));
        Fb = {-Nb * pb.y, Nb * pb.x};
      }
      C* k = row ? Krow + (hi ? W : 0) + (bx - ox) : Kcol + (hi ? TY + 2 * HALO : 0) + (by - oy);
      const bool own = unsigned(cy - oy - HALO) < unsigned(TY) && unsigned(cx - ox - HALO) < unsigned(TX);
      update_boundary<S>(out, eb, (int64_t)by * A.n[1] + bx, k, own, Fb);
    }
  }

  template <int S, bool WALLS>
  __device__ __forceinline__ void strips(const C* in, C* out, bool vec) {
    constexpr int e0 = 2 * (4 - S), RW = TX + 2 * e0;   // the stage's region
    static_assert(12 % RY == 0 && 8 % RY == 0 && 4 % RY == 0, "whole strips");
    if (WALLS && !WRAP) {
      // only the part of the region that holds interior sites (pairs and strips kept on the region's own grid)
      constexpr int R0 = HALO - e0;
      const int lx0 = max(R0, -ox), lx1 = min(R0 + RW, A.n[1] - 1 - ox);
      const int s0 = max(0, 1 - oy - R0) / RY, s1 = (min(TY + 2 * e0, A.n[0] - 1 - oy - R0) + RY - 1) / RY;
      const unsigned npair = (unsigned)(lx1 - lx0 + 1) / 2, n = npair * (unsigned)(s1 - s0);
      const unsigned inv = 0xFFFFFFFFu / npair + 1u;   // t / npair = t inv >> 32 for the few thousand t here
#pragma unroll 1
      for (unsigned t = threadIdx.x; t < n; t += NT) {
        const unsigned r = npair == 1 ? t : __umulhi(t, inv), q = t - r * npair;
        const int ly = R0 + ((int)r + s0) * RY, lx = lx0 + 2 * (int)q;
        const int gy = oy + ly, gx = ox + lx;
        strip<S, true>(in, out, ly * W + lx, S == 4 ? (int64_t)gy * A.n[1] + gx : 0, gy, gx,
                       unsigned(lx - HALO) < unsigned(TX), ly, vec);
      }
      return;
    }
    const int RH = TY + 2 * e0;
#pragma unroll 1
    for (int t = threadIdx.x; t < (RW / 2) * (RH / RY); t += NT) {
      const int r = t / (RW / 2), q = t - r * (RW / 2);
      const int ly = r * RY + HALO - e0, lx = 2 * q + HALO - e0;
      const bool own_x = unsigned(lx - HALO) < unsigned(TX);
      const int gy = oy + ly, gx = ox + lx;
      const int64_t g = S == 4 ? (int64_t)gy * A.n[1] + gx : 0;
      strip<S, WALLS>(in, out, ly * W + lx, g, gy, gx, own_x, ly, vec);
    }
  }

  // One stage from `in` to `out` (in: not const, the ghosts go into its cells beyond the walls).
  template <int S, bool WALLS>
  __device__ __forceinline__ void whole(C* in, C* out, bool vec) {
    const bool walls = WALLS && !WRAP;
    if (ORDER == 4 && walls) {
      ghosts<S>(in);
      __syncthreads();
    }
    strips<S, WALLS>(in, out, vec);
    if (walls) {
      if (S < 4) __syncthreads();   // after the strips' own writes to the boundary cells
      boundary<S>(in, out);
    }
    if (S < 4) __syncthreads();
  }

  template <bool WALLS>
  __device__ __forceinline__ void stages() {
    // 16-byte stores of Psi^{n+1} where rows and buffer allow
    const bool vec = sizeof(M) == 8 ? (A.n[1] % 2 == 0 && (uintptr_t)A.out % 16 == 0) : true;
    whole<1, WALLS>(P, a, vec);
    whole<2, WALLS>(a, b, vec);
    whole<3, WALLS>(b, a, vec);
    whole<4, WALLS>(a, b, vec);
  }

  __device__ __forceinline__ void run() {
    load();
    // a tile whose first-stage region lies two or more cells from every wall needs no wall logic
    const bool deep = ox >= 0 && ox + W <= A.n[1] && oy >= 0 && oy + TY + 2 * HALO <= A.n[0];
    if (deep) stages<false>();
    else stages<true>();
  }
};

// Tiles of a run along each axis: the interior sites [1, N-2] (periodic: every site) from coordinate 0 on.
inline void step2_tiles(int ny, int nx, bool periodic, int tx, int ty, int* ntx, int* nty) {
  const int ex = periodic ? nx : nx - 1, ey = periodic ? ny : ny - 1;
  *ntx = (ex + tx - 1) / tx;
  *nty = (ey + ty - 1) / ty;
}

}  // namespace nlse
