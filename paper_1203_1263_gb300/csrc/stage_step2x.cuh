// A whole RK4 step of a 2D FP64 grid in one launch, exact-sum stencil.
//
// As stage_step2d.cuh: a CTA takes a TX-column tile with an eight-cell halo
// through the four stages in shared memory, ghost cells beyond the walls and one
// thread per boundary site.  The tile holds every stage's input twice, in FP64
// (the pointwise terms) and as the 64-bit fixed point that the stencil sums are
// formed in, converted once where a stage produces it.  What bounds it is the
// FP64 pipe, eleven instructions per evaluated site and stage, of which the halo
// adds 1.4-2.2 times; so it pays while a step is launches and latency, and the
// stage-streaming kernels keep the larger grids (step2x_path in api.cu).
//
// The fixed-point scale of a step follows from the largest exponent of its
// Psi^n, which the step before left in a word of its own (four words in turn:
// one read, one collected, one cleared for the step after next).
#pragma once
#include "stage_step2d.cuh"

namespace nlse {

struct Step2xArgs {
  int n[2];
  int bc;
  double s, h2_over_a, cL, tiny, cLF, invcLF, sG, mL;   // as in Field
  double dtc[4];               // dt/2, dt/2, dt, dt/6, times cLF
  const double *V, *Vs;        // V and V / cLF, or nullptr
  const double2* in;
  double2* out;
  unsigned int* flag;
  unsigned int* expo;          // the four words
  int turn;                    // this step's (0..3)
  int F0, fix_offset;          // as k_fix_update
};

inline size_t step2x_smem(int tx, int ty, bool with_v) {
  const size_t W = tx + 2 * kStepHalo, H = ty + 2 * kStepHalo;
  return 5 * W * H * 16 + 2 * W * H * 2 + ((size_t)tx * ty + 2 * (W + H)) * 16 + (with_v ? 2 * W * H * 8 : 0);
}

// A site's operands in the tile: FP64 values and fixed point.
template <int W>
struct TileAccX2 {
  const double2* d;
  const longlong2* x;
  int o, F;
  __device__ __forceinline__ static int off(int k, int s) { return k == 0 ? s * W : s; }
  __device__ __forceinline__ double2 at0() const { return d[o]; }
  __device__ __forceinline__ double2 at1(int k, int s) const { return d[o + off(k, s)]; }
  __device__ __forceinline__ double2 at2(int k, int s, int j, int t) const { return d[o + off(k, s) + off(j, t)]; }
  __device__ __forceinline__ longlong2 fx0() const { return x[o]; }
  __device__ __forceinline__ longlong2 fx1(int k, int s) const { return x[o + off(k, s)]; }
  __device__ __forceinline__ longlong2 fx2(int k, int s, int j, int t) const { return x[o + off(k, s) + off(j, t)]; }
  __device__ __forceinline__ int fixF() const { return F; }
};

template <int ORDER, int TX, int NT>
struct Step2xTile {
  static constexpr int HALO = kStepHalo, W = TX + 2 * HALO;
  const Step2xArgs& A;
  const int TY, PS;
  double2 *P, *Y0, *Y1;        // Psi^n and the stage buffers, FP64
  longlong2 *X0, *X1;          // fixed point of the stage input and output, in turn
  double2 *K, *Krow, *Kcol;    // K_tot on the tile, at the boundary sites of the y and x walls
  double *V, *Vs;
  char2 *L0, *L1;              // what the fixed point of X0, X1 left out (fix_low)
  int ox, oy, F, eadj;
  bool with_v;
  unsigned int ex = 0;

  __device__ __forceinline__ Step2xTile(const Step2xArgs& A_, int rows, int tx, int ty, unsigned char* smem)
      : A(A_), TY(rows), PS(W * (rows + 2 * HALO)) {
    const int H = TY + 2 * HALO;
    P = reinterpret_cast<double2*>(smem);
    Y0 = P + PS;
    Y1 = Y0 + PS;
    X0 = reinterpret_cast<longlong2*>(Y1 + PS);
    X1 = X0 + PS;
    K = reinterpret_cast<double2*>(X1 + PS);
    Krow = K + TX * TY;
    Kcol = Krow + 2 * W;
    V = reinterpret_cast<double*>(Kcol + 2 * H);
    Vs = V + PS;
    L0 = reinterpret_cast<char2*>(with_v_of(A_) ? Vs + PS : V);
    L1 = L0 + PS;
    ox = tx * TX - HALO;
    oy = ty * TY - HALO;
    with_v = A.V != nullptr;
  }

  __device__ __forceinline__ static bool with_v_of(const Step2xArgs& a) { return a.V != nullptr; }
  __device__ __forceinline__ static char2 low(double2 v, int F) {
    return make_char2((signed char)fix_low(v.x, F), (signed char)fix_low(v.y, F));
  }
  __device__ __forceinline__ int64_t grid_index(int r, int q) const {   // of tile element (r, q); -1 outside
    int gy = oy + r, gx = ox + q;
    if (A.bc == BC_PERIODIC) {
      gy = ((gy % A.n[0]) + A.n[0]) % A.n[0];
      gx = ((gx % A.n[1]) + A.n[1]) % A.n[1];
    }
    return gy >= 0 && gy < A.n[0] && gx >= 0 && gx < A.n[1] ? (int64_t)gy * A.n[1] + gx : -1;
  }
  template <class F_>
  __device__ __forceinline__ void rows(F_&& f) const {   // f(element, grid index), a warp per row
    const int H = TY + 2 * HALO;
    for (int r = threadIdx.x >> 5; r < H; r += NT / 32)
#pragma unroll
      for (int q0 = 0; q0 < W; q0 += 32) {
        const int q = q0 + (threadIdx.x & 31);
        if (q < W) f(r * W + q, grid_index(r, q));
      }
  }
  __device__ __forceinline__ void load_potential() {
    if (with_v)
      rows([&](int e, int64_t g) {
        Step2Tile<P32, ORDER, TX, NT, 2, false>::template copy_async<8>(smem_addr(V + e), A.V + (g < 0 ? 0 : g), g < 0 ? 0 : 8);
        Step2Tile<P32, ORDER, TX, NT, 2, false>::template copy_async<8>(smem_addr(Vs + e), A.Vs + (g < 0 ? 0 : g), g < 0 ? 0 : 8);
      });
  }
  __device__ __forceinline__ static uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
  }
  __device__ __forceinline__ void load() {
    rows([&](int e, int64_t g) {
      Step2Tile<P32, ORDER, TX, NT, 2, false>::template copy_async<16>(smem_addr(P + e), A.in + (g < 0 ? 0 : g), g < 0 ? 0 : 16);
    });
    const unsigned int E = *(volatile const unsigned int*)(A.expo + A.turn);   // after grid_wait()
    F = (E > 0u && E < 2047u ? 1077 - int(E) : A.F0) + A.fix_offset;
    eadj = A.F0 - F;
    if (blockIdx.x == 0 && threadIdx.x == 0) A.expo[(A.turn + 2) & 3] = 0u;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int e = threadIdx.x; e < PS; e += NT) {
      X0[e] = fix2(P[e], F);
      L0[e] = low(P[e], F);
    }
    __syncthreads();
  }

  __device__ __forceinline__ Field<L64> field() const {
    Field<L64> f;
    f.n[0] = A.n[0]; f.n[1] = A.n[1];
    f.st[0] = W; f.st[1] = 1;
    f.s = A.s;
    f.h2_over_a = A.h2_over_a;
    f.cL = A.cL;
    f.tiny = A.tiny;
    f.bc = A.bc;
    f.F = A.F0;
    f.cLF = A.cLF;
    f.invcLF = A.invcLF;
    f.sG = A.sG;
    f.V = with_v ? reinterpret_cast<const OnChip<double>*>(V) : nullptr;
    return f;
  }

  // F in units of cLF at element e (grid site idx), every stencil operand in the tile (a_lap_exact's sums, the
  // ghosts in their cells).
  __device__ __forceinline__ double2 rhs(const double2* d, const longlong2* x, const char2* l, int e, int gy, int gx) const {
    const double2 pc = d[e];
    const longlong2 cc = x[e], xm = x[e - 1], xp = x[e + 1], ym = x[e - W], yp = x[e + W];
    bool bad = fbad(cc) | fbad(xm) | fbad(xp) | fbad(ym) | fbad(yp);
    long long sx = (yp.x + ym.x) + (xp.x + xm.x), sy = (yp.y + ym.y) + (xp.y + xm.y);
    int rx, ry;
    const char2 lc = l[e], l0 = l[e - 1], l1 = l[e + 1], l2 = l[e - W], l3 = l[e + W];   // fix_correction
    if constexpr (ORDER == 4) {
      const longlong2 xm2 = x[e - 2], xp2 = x[e + 2], ym2 = x[e - 2 * W], yp2 = x[e + 2 * W];
      bad |= fbad(xm2) | fbad(xp2) | fbad(ym2) | fbad(yp2);
      sx = 16 * sx - ((ym2.x + yp2.x) + (xm2.x + xp2.x)) - 60 * cc.x;
      sy = 16 * sy - ((ym2.y + yp2.y) + (xm2.y + xp2.y)) - 60 * cc.y;
      const char2 m0 = l[e - 2], m1 = l[e + 2], m2 = l[e - 2 * W], m3 = l[e + 2 * W];
      rx = 16 * ((l0.x + l1.x) + (l2.x + l3.x)) - ((m0.x + m1.x) + (m2.x + m3.x)) - 60 * lc.x;
      ry = 16 * ((l0.y + l1.y) + (l2.y + l3.y)) - ((m0.y + m1.y) + (m2.y + m3.y)) - 60 * lc.y;
    } else {
      sx -= 4 * cc.x;
      sy -= 4 * cc.y;
      rx = (l0.x + l1.x) + (l2.x + l3.x) - 4 * lc.x;
      ry = (l0.y + l1.y) + (l2.y + l3.y) - 4 * lc.y;
    }
    const double N = fma(A.sG, norm2(pc), -(with_v ? Vs[e] : 0.0));
    double2 aL;
    if (!bad) {
      aL = {__dmul_rn(A.mL, i2d_low(sx, rx, eadj)), __dmul_rn(A.mL, i2d_low(sy, ry, eadj))};
    } else {   // an operand out of the fixed-point range: the FP64 stencil
      const Field<L64> f = field();
      TileAccX2<W> acc{d, x, e, F};
      const int idx[2] = {gy, gx};
      const double Nc = __dmul_rn(N, A.cLF);   // as in a_lap_exact
      if (A.bc != BC_PERIODIC) aL = a_lap_body<L64, 2, ORDER, TileAccX2<W>, true>(f, acc, idx, e, pc, Nc);
      else aL = a_lap_body<L64, 2, ORDER, TileAccX2<W>, false>(f, acc, idx, e, pc, Nc);
      aL = {aL.x * A.invcLF, aL.y * A.invcLF};
    }
    return {-fma(N, pc.y, aL.y), fma(N, pc.x, aL.x)};
  }

  // The stage's update of element e with K_tot at k (own sites), the result into d / x (stages 1-3) or Psi^{n+1}.
  __device__ __forceinline__ void update(int S, double2* d, longlong2* x, char2* l, int e, int64_t g, double2* k, bool own,
                                         double2 Fv) {
    if (S < 4) {
      if (own) {
        if (S == 1) *k = Fv;
        else *k = double2{fma(2.0, Fv.x, k->x), fma(2.0, Fv.y, k->y)};
      }
      const double2 pn = P[e];
      const double2 y = {fma(A.dtc[S - 1], Fv.x, pn.x), fma(A.dtc[S - 1], Fv.y, pn.y)};
      d[e] = y;
      x[e] = fix2(y, F);
      l[e] = low(y, F);
    } else if (own) {
      const double2 pn = P[e], kt = *k;
      const double2 q = {fma(A.dtc[3], kt.x + Fv.x, pn.x), fma(A.dtc[3], kt.y + Fv.y, pn.y)};
      A.out[g] = q;
      if (!(finite_bits(q.x) && finite_bits(q.y))) atomicOr(A.flag, 1u);
      ex = max(ex, max(range_bits(q.x), range_bits(q.y)));
    }
  }

  struct Clip { int ylo, yhi, xlo, xhi; bool top, bot, left, right; };
  __device__ __forceinline__ Clip clip(int S) const {   // the stage's interior sites, clipped to the grid (walls)
    const int e0 = 2 * (4 - S);
    Clip c;
    const int b = A.bc == BC_PERIODIC ? 0 : 1;
    // a periodic grid's last tiles overhang: their stages 1-3 go on past the end, stage 4 does not
    c.ylo = A.bc == BC_PERIODIC ? oy + HALO - e0 : max(oy + HALO - e0, b);
    c.xlo = A.bc == BC_PERIODIC ? ox + HALO - e0 : max(ox + HALO - e0, b);
    c.yhi = oy + HALO + TY + e0;
    c.xhi = ox + HALO + TX + e0;
    if (b || S == 4) {
      c.yhi = min(c.yhi, A.n[0] - b);
      c.xhi = min(c.xhi, A.n[1] - b);
    }
    c.top = b && c.ylo == 1;
    c.bot = b && c.yhi == A.n[0] - 1;
    c.left = b && c.xlo == 1;
    c.right = b && c.xhi == A.n[1] - 1;
    return c;
  }

  __device__ __forceinline__ void ghosts(const Clip& c, const double2* d, longlong2* x, char2* l) {
    const Field<L64> f = field();
    const int rw = c.xhi - c.xlo, rh = c.yhi - c.ylo;
    const int n0 = c.top ? rw : 0, n1 = n0 + (c.bot ? rw : 0), n2 = n1 + (c.left ? rh : 0), n3 = n2 + (c.right ? rh : 0);
#pragma unroll 1
    for (int t = threadIdx.x; t < n3; t += NT) {
      const bool row = t < n1, hi = row ? t >= n0 : t >= n2;
      const int gy = row ? (hi ? A.n[0] - 2 : 1) : c.ylo + (t - (hi ? n2 : n1));
      const int gx = row ? c.xlo + (t - (hi ? n0 : 0)) : (hi ? A.n[1] - 2 : 1);
      const int e = (gy - oy) * W + (gx - ox), dir = hi ? 1 : -1;
      TileAccX2<W> acc{d, x, e, F};
      const double2 pc = d[e];
      const longlong2 cc = x[e], u = x[e + W], w = x[e - W], p = x[e + 1], m = x[e - 1];
      double2 dh = {0.0, 0.0};
      double Nc = 0.0, m2 = 0.0;
      if (A.bc == BC_MSD) {   // only the MSD wall's form takes these
        const double nn = norm2(pc);
        m2 = nn > A.tiny ? nn : 0.0;
        Nc = __dmul_rn(fma(A.sG, nn, -(with_v ? Vs[e] : 0.0)), A.cLF);
        dh = {i2d_rn((u.x + w.x) + (p.x + m.x) - 4 * cc.x, -F), i2d_rn((u.y + w.y) + (p.y + m.y) - 4 * cc.y, -F)};
      }
      bool bad = false;
      longlong2 g;
      if (row) g = ghost_fix<L64, 2>(f, acc, 0, dir, e, pc, dh, Nc, m2, F, &bad);
      else g = ghost_fix<L64, 2>(f, acc, 1, dir, e, pc, dh, Nc, m2, F, &bad);
      x[e + 2 * dir * (row ? W : 1)] = bad ? longlong2{kFixBad, kFixBad} : g;
      l[e + 2 * dir * (row ? W : 1)] = make_char2(0, 0);
    }
  }

  __device__ __forceinline__ void boundary(int S, const Clip& c, const double2* din, const longlong2* xin, const char2* lin,
                                           double2* dout, longlong2* xout, char2* lout) {
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
      double2 Fb = {0.0, 0.0};
      if (A.bc == BC_MSD) {
        const int e = (cy - oy) * W + (cx - ox);
        const double2 pc = din[e], pb = din[eb];
        const double2 Fv = rhs(din, xin, lin, e, cy, cx);
        const double m2 = norm2(pc);
        double theta = 0.0;
        if (m2 > A.tiny) theta = fma(Fv.y, pc.x, -(Fv.x * pc.y)) / m2;
        Fb = {-theta * pb.y, theta * pb.x};
      } else if (A.bc == BC_L0) {
        const double2 pb = din[eb];
        const double Nb = fma(A.sG, norm2(pb), -(with_v ? Vs[eb] : 0.0));
        Fb = {-Nb * pb.y, Nb * pb.x};
      }
      double2* k = row ? Krow + (hi ? W : 0) + (bx - ox) : Kcol + (hi ? TY + 2 * HALO : 0) + (by - oy);
      const bool own = unsigned(cy - oy - HALO) < unsigned(TY) && unsigned(cx - ox - HALO) < unsigned(TX);
      if (S < 4 || own) update(S, dout, xout, lout, eb, (int64_t)by * A.n[1] + bx, k, true, Fb);
    }
  }

  __device__ __forceinline__ void run() {
    load();
    const bool walls = A.bc != BC_PERIODIC &&
                       !(ox >= 0 && ox + W <= A.n[1] && oy >= 0 && oy + TY + 2 * HALO <= A.n[0]);
    const double2* din = P;
    double2 *dout = Y0, *dnext = Y1;
    longlong2 *xin = X0, *xout = X1;
    char2 *lin = L0, *lout = L1;
    // one body for the four stages: a step is short enough that fetching its instructions counts
#pragma unroll 1
    for (int S = 1; S <= 4; ++S) {
      const Clip c = clip(S);
      if (ORDER == 4 && walls) {
        ghosts(c, din, xin, lin);
        __syncthreads();
      }
      const unsigned rw = (unsigned)(c.xhi - c.xlo), n = rw * (unsigned)(c.yhi - c.ylo);
      const unsigned inv = 0xFFFFFFFFu / rw + 1u;   // t / rw for the few thousand t here
#pragma unroll 1
      for (unsigned t = threadIdx.x; t < n; t += NT) {
        const unsigned r = rw == 1 ? t : __umulhi(t, inv), q = t - r * rw;
        const int gy = c.ylo + (int)r, gx = c.xlo + (int)q, ly = gy - oy, lx = gx - ox, e = ly * W + lx;
        const double2 Fv = rhs(din, xin, lin, e, gy, gx);
        const bool own = unsigned(ly - HALO) < unsigned(TY) && unsigned(lx - HALO) < unsigned(TX);
        update(S, dout, xout, lout, e, (int64_t)gy * A.n[1] + gx, K + ((ly - HALO) * TX + lx - HALO), own, Fv);
      }
      if (walls) boundary(S, c, din, xin, lin, dout, xout, lout);
      __syncthreads();
      din = dout;
      double2* d = dout;
      dout = dnext;
      dnext = d;
      char2* l = lin;
      lin = lout;
      lout = l;
      longlong2* x = xin;
      xin = xout;
      xout = x;
    }
    emax_commit(A.expo + ((A.turn + 1) & 3), ex);
  }
};

}  // namespace nlse
