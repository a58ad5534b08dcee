// The C ABI of include/nlse.h: argument checks, workspace layout, stage
// dispatch, CUDA-graph chunking of the step loop, reductions and errors.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>
#include <string>

#include "../../include/nlse.h"
#include "nlse_internal.h"
#include "stage_march.cuh"

using namespace nlse;

namespace {

thread_local char g_err[512] = "";

int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}

int cuda_fail(cudaError_t e, const char* where) {
  return fail(NLSE_ECUDA, "%s: %s", where, cudaGetErrorString(e));
}

constexpr int kGraphSteps = 16;   // RK4 steps captured per graph replay
constexpr long long kSpinLimit = 2000000000ll;   // ~1 s of SM clock: bound on device-side waits
constexpr unsigned int kFlagTimeoutBit = 4u;

// cuTensorMapEncodeTiled, resolved once through the runtime (no link to libcuda).
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    else
      cudaGetLastError();
  }
  return fn;
}
constexpr size_t kAlign = 256;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct Layout {
  size_t ktot, ptmp, pout, pn32, vs, alt, partials, status, total;
};

bool layout_for(int dims, const int64_t* N, int dtype, Layout* L, int64_t* total_sites) {
  if (dims < 1 || dims > 3 || !N) return false;
  if (dtype < NLSE_C128 || dtype > NLSE_C64_ACC64) return false;
  int64_t total = 1;
  for (int k = 0; k < dims; ++k) {
    if (N[k] < 3 || N[k] > (int64_t(1) << 30)) return false;
    total *= N[k];
    if (total > (int64_t(1) << 40)) return false;
  }
  const size_t es = (dtype == NLSE_C128) ? 16 : 8;
  size_t off = 0;
  L->ktot = off; off = align_up(off + es * total);
  L->ptmp = off; off = align_up(off + es * total);
  L->pout = off; off = align_up(off + es * total);
  L->pn32 = off; if (dtype == NLSE_C64_ACC64) off = align_up(off + 8 * total);
  L->vs = off; if (dtype == NLSE_C128) off = align_up(off + 8 * total);   // V / cLF for the exact-sum stages
  L->alt = off; if (dtype == NLSE_C64 && dims == 3) off = align_up(off + 8 * total);   // Psi ping-pong (fused step)
  L->partials = off; off = align_up(off + sizeof(double) * 2 * kMaxReduceBlocks);
  L->status = off; off = align_up(off + 256);
  L->total = off;
  if (total_sites) *total_sites = total;
  return true;
}

}  // namespace

struct nlse_ctx {
  int d;
  int64_t n[3];
  int64_t total;
  double h, a, s;
  int bc, order, dtype;
  void* psi;
  const void* V;
  cudaStream_t stream;
  char* ws;
  Layout lay;
  double vmax;
  int fixF;          // reference fraction bits F0 of the exact-sum stencil (FP64 path): cLF = cL 2^-F0
  int fix_offset;    // test hook added to the derived fraction bits (nlse_debug_set)
  int variant, tile_cfg;
  bool chosen;       // the caller chose the variant (nlse_set_kernel)
  cudaStream_t cap;
  cudaGraphExec_t exec;
  double graph_dt;
  int graph_variant;
  // TMA descriptors of the stage inputs (Psi or its FP32 copy, Psi_tmp, Psi_out) per tile shape
  CUtensorMap tmaps[4][3];
  signed char tmap_state[4][3];   // 0 = not built, 1 = ok, -1 = layout not eligible
  CUtensorMap fmaps[3];           // the fused kernel's inputs: Psi, its ping-pong copy, Psi_out
  signed char fmap_state[3];
  long long spin_limit;           // bound on device-side waits (cycles)
  unsigned int extra_tx;          // test hook, see nlse_debug_set
  bool line_failed;               // the 1D cluster path could not be launched here: per-site kernel instead
  cudaStream_t side;              // wall-shell kernels run here, concurrently with the deep kernels
  cudaEvent_t ev_fork, ev_join;
  cudaStream_t side_yx[2];        // 3D: the y- and x-wall slabs' streams
  cudaEvent_t ev_join_yx[2];

  void* at(size_t off) const { return ws + off; }
  unsigned int* flag() const { return (unsigned int*)(ws + lay.status); }
  unsigned long long* vbits() const { return (unsigned long long*)(ws + lay.status + 8); }
  int* fdev() const { return (int*)(ws + lay.status + 16); }                    // current fraction bits
  unsigned int* emax() const { return (unsigned int*)(ws + lay.status + 20); }  // stage-4 largest exponent
  bool exact() const { return dtype == NLSE_C128 && variant >= 2 && variant <= 3; }
  unsigned int* expo() const { return (unsigned int*)(ws + lay.status + 40); }  // the whole-step kernel's four words
  unsigned int* done() const { return (unsigned int*)(ws + lay.status + 32); }  // blocks of a reduction that are through
  double* result() const { return (double*)(ws + lay.status + 64); }
  double* partials() const { return (double*)(ws + lay.partials); }
};

namespace {

// Tile shape in use: the caller's choice, else the measured default per form
// and size (nlse_autotune can refine it): 32x8 for FP64; for the FP32 forms
// in 3D, where the tiles serve them (above 3,000,000 sites, and periodic grids),
// 64x8 on planes of at least 8192 sites (fewer, wider TMA boxes; FP32 512x256x256
// 953 against 996 us per step with 32x8, periodic 128^3 70.2 against 72.8) and
// 32x8 on smaller planes (enough CTAs to fill the SMs; periodic 80^3 37.8 against
// 41.0, 88^3 41.5 against 46.9); 32x16 in 2D (F of large periodic planes).
int resolved_tile(const nlse_ctx* c) {
  if (c->tile_cfg >= 0) return c->tile_cfg;
  if (c->dtype == NLSE_C128) return 0;
  if (c->d == 3) return c->n[1] * c->n[2] >= 8192 ? 3 : 0;
  return 2;
}

template <class T>
Field<T> make_field(const nlse_ctx* c, const void* in) {
  using R = typename T::R;
  Field<T> f;
  memset(&f, 0, sizeof(f));
  for (int k = 0; k < 3; ++k) { f.n[k] = 1; f.m[k] = 1; f.st[k] = 0; }
  int64_t stride = 1;
  for (int k = c->d - 1; k >= 0; --k) {
    f.n[k] = int(c->n[k]);
    f.m[k] = int(c->n[k] - 2);
    f.st[k] = stride;
    stride *= c->n[k];
  }
  f.ninterior = 1;
  for (int k = 0; k < c->d; ++k) f.ninterior *= (c->n[k] - 2);
  f.a = R(c->a);
  f.s = R(c->s);
  f.h2_over_a = R(c->h * c->h / c->a);
  f.cL = R(c->order == 4 ? c->a / (12.0 * c->h * c->h) : c->a / (c->h * c->h));
  f.tiny = R(sizeof(R) == 8 ? 1e-300 : 1e-30);
  f.bc = c->bc;
  f.F = c->fixF;
  f.Fdev = (c->dtype == NLSE_C128) ? c->fdev() : nullptr;
  f.fine = c->d == 2 && step2x_fits(int(c->n[0]), int(c->n[1]), c->bc == NLSE_BC_PERIODIC);
  const double cL = c->order == 4 ? c->a / (12.0 * c->h * c->h) : c->a / (c->h * c->h);
  int ex = 0;
  f.mL = 2.0 * frexp(cL, &ex);
  f.cLF = f.fine ? ldexp(0.5, ex - c->fixF) : ldexp(cL, -c->fixF);
  f.invcLF = R(1.0 / f.cLF);
  f.sG = R(c->s / f.cLF);
  f.V = (const typename T::VR*)c->V;
  f.in = (const typename T::C*)in;
  return f;
}

LaunchCfg launch_cfg(const nlse_ctx* c);

template <class T>
cudaError_t dispatch_stage(const nlse_ctx* c, const StageArgs<T>& A, const void* tmap, cudaStream_t st, int variant = -1) {
  LaunchCfg L = launch_cfg(c);
  if (variant < 0) variant = c->variant;
  L.variant = (variant == 4) ? 1 : variant;   // single stages of the fused variant: the tiled kernel
  L.tmap = tmap;
  switch (c->d * 10 + c->order) {
    case 12: return launch_stage<T, 1, 2>(A, L, st);
    case 14: return launch_stage<T, 1, 4>(A, L, st);
    case 22: return launch_stage<T, 2, 2>(A, L, st);
    case 24: return launch_stage<T, 2, 4>(A, L, st);
    case 32: return launch_stage<T, 3, 2>(A, L, st);
    default: return launch_stage<T, 3, 4>(A, L, st);
  }
}

// A 3D TMA descriptor over a complex field of the context's shape (real components of es bytes) with a
// box of box_x components by box_y rows by one plane; false when the layout is not eligible (TMA needs
// 16-byte row pitches and a 16-byte aligned base).
bool encode_field_map(const nlse_ctx* c, CUtensorMap* m, const void* ptr, size_t es, int box_x, int box_y) {
  const cuuint64_t nx = c->n[2], ny = c->n[1], nz = c->n[0];
  EncodeTiledFn fn = encode_fn();
  if (!fn || (2 * nx * es) % 16 != 0 || ((uintptr_t)ptr % 16) != 0) return false;
  cuuint64_t dims[3] = {2 * nx, ny, nz};
  cuuint64_t strides[2] = {2 * nx * es, 2 * nx * ny * es};
  cuuint32_t box[3] = {cuuint32_t(box_x), cuuint32_t(box_y), 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, es == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(ptr),
            dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The fused kernel's TMA descriptor of buffer `buf` (0 = Psi, 1 = its ping-pong copy, 2 = Psi_out).
const CUtensorMap* fused_tmap(const nlse_ctx* cc, int buf, const void* ptr) {
  nlse_ctx* c = const_cast<nlse_ctx*>(cc);
  signed char& st = c->fmap_state[buf];
  if (st == 0) st = encode_field_map(c, &c->fmaps[buf], ptr, 4, kFusedBoxX, kFusedBoxY) ? 1 : -1;
  return st == 1 ? &c->fmaps[buf] : nullptr;
}

// The fused step runs for the FP32 form on 3D grids with every extent >= 16
// and TMA-eligible rows, except on periodic grids (their shell wraps).
bool fused_path(const nlse_ctx* c) {
  if (c->variant != 4 || c->dtype != NLSE_C64 || c->d != 3 || c->bc == NLSE_BC_PERIODIC) return false;
  const int n[3] = {int(c->n[0]), int(c->n[1]), int(c->n[2])};
  if (!fused_grid_ok(3, n)) return false;
  return fused_tmap(c, 0, c->psi) && fused_tmap(c, 1, c->at(c->lay.alt)) && fused_tmap(c, 2, c->at(c->lay.pout));
}

// The TMA descriptor of stage-input buffer `buf` (0 = Psi or its FP32 copy,
// 1 = Psi_tmp, 2 = Psi_out) for the 3D tiled kernel's tile, or nullptr when
// the layout is not eligible (TMA needs 16-byte row pitches).
const CUtensorMap* stage_tmap(const nlse_ctx* cc, int buf, const void* ptr) {
  nlse_ctx* c = const_cast<nlse_ctx*>(cc);
  if (c->d != 3 || (c->variant != 1 && c->variant != 2 && c->variant != 4)) return nullptr;
  const int tc = resolved_tile(c);
  signed char& st = c->tmap_state[tc][buf];
  if (st == 0) {
    st = -1;
    int tx, ty;
    tma_tile_shape(tc, &tx, &ty);
    const size_t es = (c->dtype == NLSE_C128) ? 8 : 4;   // bytes of one real component
    const cuuint64_t nx = c->n[2], ny = c->n[1], nz = c->n[0];
    EncodeTiledFn fn = encode_fn();
    if (fn && (2 * nx * es) % 16 == 0 && ((uintptr_t)ptr % 16) == 0) {
      cuuint64_t dims[3] = {2 * nx, ny, nz};
      cuuint64_t strides[2] = {2 * nx * es, 2 * nx * ny * es};
      cuuint32_t box[3] = {cuuint32_t(2 * (tx + 4)), cuuint32_t(ty + 4), 1};
      cuuint32_t estr[3] = {1, 1, 1};
      CUresult r = fn(&c->tmaps[tc][buf], es == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3,
                      const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                      CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r == CUDA_SUCCESS) st = 1;
    }
  }
  return st == 1 ? &c->tmaps[tc][buf] : nullptr;
}

// The arguments of stage s (1..4) of Eq. RK4_GPU: Psi -> Psi_tmp -> Psi_out ->
// Psi_tmp -> Psi.  cur holds Psi^n, stage 4 writes Psi^{n+1} to nxt (the same
// buffer except on the fused path's ping-pong steps).
template <class T>
StageArgs<T> stage_args(const nlse_ctx* c, int s, double dt, void* cur, void* nxt) {
  using C = typename T::C;
  using R = typename T::R;
  const bool mix = (c->dtype == NLSE_C64_ACC64);
  C* ktot = (C*)c->at(c->lay.ktot);
  C* ptmp = (C*)c->at(c->lay.ptmp);
  C* pout = (C*)c->at(c->lay.pout);
  const C* psin = mix ? (const C*)c->at(c->lay.pn32) : (const C*)cur;
  const void* in[4] = {psin, ptmp, pout, ptmp};
  C* outs[4] = {ptmp, pout, ptmp, nullptr};
  const double dtc[4] = {dt / 2.0, dt / 2.0, dt, dt / 6.0};
  const int i = s - 1;
  StageArgs<T> A;
  memset(&A, 0, sizeof(A));
  A.f = make_field<T>(c, in[i]);
  A.psin = psin;
  A.ktot = ktot;
  A.out = outs[i];
  A.master = (typename T::M*)nxt;
  A.master_in = (const typename T::M*)cur;
  A.n32 = mix ? (C*)c->at(c->lay.pn32) : nullptr;
  // FP64 with the exact-sum stencil: F is formed in units of cLF, so the stage coefficient carries it
  const bool g = std::is_same<T, P64>::value && c->exact();
  A.dtc = R(g ? dtc[i] * A.f.cLF : dtc[i]);
  A.dt6 = dt / 6.0;
  A.stage = s;
  A.flag = c->flag();
  A.Vs = (g && c->V) ? (const typename T::VR*)c->at(c->lay.vs) : nullptr;
  A.emax = (g && s == 4) ? c->emax() : nullptr;   // collects the exponent of Psi^{n+1}
  return A;
}

// Stage s of one step, Psi updated in place.
template <class T>
cudaError_t launch_one_stage(const nlse_ctx* c, int s, double dt, cudaStream_t st) {
  const StageArgs<T> A = stage_args<T>(c, s, dt, c->psi, c->psi);
  const int inbuf[4] = {0, 1, 2, 1};
  return dispatch_stage<T>(c, A, stage_tmap(c, inbuf[s - 1], A.f.in), st);
}

LaunchCfg launch_cfg(const nlse_ctx* c) {
  LaunchCfg L;
  L.variant = c->variant;
  L.tile_cfg = resolved_tile(c);
  L.tmap = nullptr;
  L.spin_limit = c->spin_limit;
  L.extra_tx = c->extra_tx;
  L.side = c->side;
  L.ev_fork = c->ev_fork;
  L.ev_join = c->ev_join;
  for (int i = 0; i < 2; ++i) {
    L.side_yx[i] = c->side_yx[i];
    L.ev_join_yx[i] = c->ev_join_yx[i];
  }
  return L;
}

// 1D lines that take the cluster path: FP64 with the exact-sum stencil (variant 2).
bool line_path(const nlse_ctx* c) {
  return c->d == 1 && !c->line_failed && c->dtype == NLSE_C128 && c->variant == 2 && line_ok(int(c->n[0]));
}

// 1D lines that run several steps per launch: variant 1 (and what runs as it) with the FP64 stencil up to the
// length the cluster path has, with FP32 stages at any length; and FP64 lines whose default is one thread per site
// with the FP64 stencil (variant 0: the same arithmetic), up to the length where a launch per stage is the faster
// one: central differences 14,000 sites 7.2 against 9.7 us per step, 18,000 10.6 against 9.9 (MSD 22,000 11.4 and
// 12.9, 24,000 14.4 and 13.0); 2SHOC periodic 12,000 8.2 and 10.7, 16,000 13.4 and 11.0; 2SHOC between walls 32,768
// 15.0 and 19.1.
bool lines_path(const nlse_ctx* c) {
  if (c->d != 1) return false;
  if (c->dtype == NLSE_C128) {
    if (c->variant == 0) {
      const bool msd = c->bc == NLSE_BC_MSD;
      const int64_t longest = c->order == 2 ? (msd ? 22500 : 14500) : (c->bc == NLSE_BC_PERIODIC ? 12500 : int64_t(1) << 15);
      return !c->chosen && c->n[0] <= longest;
    }
    return (c->variant == 1 || c->variant == 4) && line_ok(int(c->n[0]));
  }
  return c->variant == 1 || c->variant == 2 || c->variant == 4;
}

cudaError_t launch_line(const nlse_ctx* c, int64_t nsteps, double dt) {
  StageArgs<P64> A[4];
  for (int s = 1; s <= 4; ++s) A[s - 1] = stage_args<P64>(c, s, dt, c->psi, c->psi);
  return launch_line_steps(A, nsteps, int(c->n[0]), c->order, c->fixF, c->fix_offset, c->stream);
}

// Psi's ping-pong copy on the whole-step paths: the stage arrays they do not use (K_tot; in the mixed form K_tot
// and Psi_tmp, which lie one after the other, hold the FP64 master).
void* step_alt(const nlse_ctx* c) { return c->at(c->lay.ktot); }

// The arguments that the 1D and 2D whole-step kernels share.
template <class T, class A>
A step_args(const nlse_ctx* c, double dt, const void* cur, void* nxt) {
  const Field<T> f = make_field<T>(c, cur);
  A a;
  memset(&a, 0, sizeof(a));
  a.bc = f.bc;
  a.s = f.s;
  a.h2_over_a = f.h2_over_a;
  a.cL = f.cL;
  a.tiny = f.tiny;
  const double dtc[4] = {dt / 2.0, dt / 2.0, dt, dt / 6.0};
  for (int i = 0; i < 4; ++i) a.dtc[i] = typename T::R(dtc[i]);
  a.V = f.V;
  a.in = (const typename T::M*)cur;
  a.out = (typename T::M*)nxt;
  a.flag = c->flag();
  return a;
}

int steps_per_launch(const nlse_ctx* c) {
  const int n = int(c->n[0]);
  return c->dtype == NLSE_C128 ? steps1d_per_launch<P64>(n)
                               : (c->dtype == NLSE_C64 ? steps1d_per_launch<P32>(n) : steps1d_per_launch<PMix>(n));
}

template <class T>
cudaError_t launch_steps1(const nlse_ctx* c, double dt, int steps, cudaStream_t st, const void* cur, void* nxt, bool early) {
  Step1Args<T> A = step_args<T, Step1Args<T>>(c, dt, cur, nxt);
  A.n = int(c->n[0]);
  return launch_steps1d<T>(A, c->order, steps, early, st);
}

// (early: not a call's first launch, see launch_early)
cudaError_t launch_steps1_any(const nlse_ctx* c, double dt, int steps, cudaStream_t st, const void* cur, void* nxt,
                              bool early) {
  switch (c->dtype) {
    case NLSE_C128: return launch_steps1<P64>(c, dt, steps, st, cur, nxt, early);
    case NLSE_C64: return launch_steps1<P32>(c, dt, steps, st, cur, nxt, early);
    default: return launch_steps1<PMix>(c, dt, steps, st, cur, nxt, early);
  }
}

// One step of the fused path from buffer cur to buffer nxt (Psi or its ping-pong copy).
cudaError_t launch_step_fused(const nlse_ctx* c, double dt, cudaStream_t st, void* cur, void* nxt) {
  StageArgs<P32> A[4];
  for (int s = 1; s <= 4; ++s) A[s - 1] = stage_args<P32>(c, s, dt, cur, nxt);
  const CUtensorMap* tm12 = fused_tmap(c, cur == c->psi ? 0 : 1, cur);
  const CUtensorMap* tm34 = fused_tmap(c, 2, c->at(c->lay.pout));
  const LaunchCfg L = launch_cfg(c);
  return c->order == 4 ? launch_fused_step<4>(A, tm12, tm34, L, st) : launch_fused_step<2>(A, tm12, tm34, L, st);
}

// Small 2D grids of the exact-sum stencil on the whole-step kernel.
bool step2x_path(const nlse_ctx* c) {
  return c->d == 2 && c->dtype == NLSE_C128 && c->variant == 2 &&
         step2x_fits(int(c->n[0]), int(c->n[1]), c->bc == NLSE_BC_PERIODIC);
}

// FP32 forms' 3D grids whose steps take the columns kernel: its launches do not depend on the tile.
bool columns_path(const nlse_ctx* c) {
  if (c->d != 3 || c->dtype == NLSE_C128 || c->extra_tx) return false;
  const Field<P32> f = make_field<P32>(c, c->psi);
  const void* in = c->dtype == NLSE_C64_ACC64 ? c->at(c->lay.pn32) : c->psi;
  const bool tma = stage_tmap(c, 0, in) != nullptr;
  return c->order == 4 ? march_serves<4>(f, tma) : march_serves<2>(f, tma);
}

// The FP32 forms' 2D grids on the whole-step kernel (the tiled variants); not the mixed form's long periodic planes of
// three or four rows, whose tiles would be mostly wrapped halo, each row of it rounded from the FP64 master (3x20000
// 11.9 us per step, one thread per site 9.4; 3x4800 5.5 and 9.8).
bool step2_path(const nlse_ctx* c) {
  if (c->dtype == NLSE_C64_ACC64 && c->bc == NLSE_BC_PERIODIC && c->n[0] < 5 && c->n[1] > 12000) return false;
  return c->d == 2 && c->dtype != NLSE_C128 && (c->variant == 1 || c->variant == 2 || c->variant == 4);
}

template <class T>
cudaError_t launch_step2(const nlse_ctx* c, double dt, cudaStream_t st, const void* cur, void* nxt, bool early) {
  Step2Args<T> A = step_args<T, Step2Args<T>>(c, dt, cur, nxt);
  A.n[0] = int(c->n[0]);
  A.n[1] = int(c->n[1]);
  return launch_step2d<T>(A, c->order, c->tile_cfg, early, st);
}

cudaError_t launch_step2x_any(const nlse_ctx* c, double dt, cudaStream_t st, const void* cur, void* nxt, int turn,
                              bool early) {
  const Field<P64> f = make_field<P64>(c, cur);
  Step2xArgs A = step_args<P64, Step2xArgs>(c, dt, cur, nxt);
  A.n[0] = int(c->n[0]);
  A.n[1] = int(c->n[1]);
  A.cLF = f.cLF;
  A.invcLF = f.invcLF;
  A.mL = f.mL;
  A.sG = f.sG;
  for (int i = 0; i < 4; ++i) A.dtc[i] = A.dtc[i] * f.cLF;
  A.Vs = c->V ? (const double*)c->at(c->lay.vs) : nullptr;
  A.expo = c->expo();
  A.turn = turn & 3;
  A.F0 = c->fixF;
  A.fix_offset = c->fix_offset;
  return launch_step2x(A, c->order, early, st);
}

// Step i of a run of steps (the first one an ordinary launch).
cudaError_t launch_step2_any(const nlse_ctx* c, double dt, cudaStream_t st, const void* cur, void* nxt, int i) {
  switch (c->dtype) {
    case NLSE_C128: return launch_step2x_any(c, dt, st, cur, nxt, i, i > 0);
    case NLSE_C64: return launch_step2<P32>(c, dt, st, cur, nxt, i > 0);
    default: return launch_step2<PMix>(c, dt, st, cur, nxt, i > 0);
  }
}

// The exact-sum stencil's scale for the next step: from the exponent stage 4
// collected (psi == nullptr) or from a full pass over psi.
cudaError_t update_fix(const nlse_ctx* c, const void* psi, cudaStream_t st) {
  return launch_fix_update((const double*)psi, 2 * c->total, c->emax(), c->fdev(), c->fixF, c->fix_offset, st);
}

template <class T>
cudaError_t launch_step(const nlse_ctx* c, double dt, cudaStream_t st) {
  for (int s = 1; s <= 4; ++s) {
    cudaError_t e = launch_one_stage<T>(c, s, dt, st);
    if (e != cudaSuccess) return e;
  }
  if (std::is_same<T, P64>::value && c->exact()) return update_fix(c, nullptr, st);
  return cudaSuccess;
}

cudaError_t launch_stage_any(const nlse_ctx* c, int s, double dt, cudaStream_t st) {
  switch (c->dtype) {
    case NLSE_C128: return launch_one_stage<P64>(c, s, dt, st);
    case NLSE_C64: return launch_one_stage<P32>(c, s, dt, st);
    default: return launch_one_stage<PMix>(c, s, dt, st);
  }
}

cudaError_t launch_step_any(const nlse_ctx* c, double dt, cudaStream_t st) {
  switch (c->dtype) {
    case NLSE_C128: return launch_step<P64>(c, dt, st);
    case NLSE_C64: return launch_step<P32>(c, dt, st);
    default: return launch_step<PMix>(c, dt, st);
  }
}

void drop_graph(nlse_ctx* c) {
  if (c->exec) cudaGraphExecDestroy(c->exec);
  c->exec = nullptr;
}

int ensure_graph(nlse_ctx* c, double dt) {
  if (c->exec && c->graph_dt == dt) return NLSE_OK;
  drop_graph(c);
  if (!c->cap) {
    cudaError_t e = cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_fail(e, "cudaStreamCreate");
  }
  cudaError_t e = cudaStreamBeginCapture(c->cap, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamBeginCapture");
  cudaError_t le = cudaSuccess;
  const bool fused = fused_path(c), step2 = step2_path(c) || step2x_path(c), lines = lines_path(c);
  const int per = lines ? steps_per_launch(c) : 1;   // divides kGraphSteps an even number of times
  for (int i = 0; i < kGraphSteps / per && le == cudaSuccess; ++i) {
    if (lines) {   // ping-pong as below
      void* a = c->psi;
      void* b = step_alt(c);
      le = (i % 2 == 0) ? launch_steps1_any(c, dt, per, c->cap, a, b, i > 0)
                        : launch_steps1_any(c, dt, per, c->cap, b, a, true);
    } else if (step2) {
      void* a = c->psi;
      void* b = step_alt(c);
      le = (i % 2 == 0) ? launch_step2_any(c, dt, c->cap, a, b, i) : launch_step2_any(c, dt, c->cap, b, a, i);
    } else if (fused) {   // ping-pong: even steps Psi -> copy, odd steps copy -> Psi (kGraphSteps is even)
      void* a = c->psi;
      void* b = c->at(c->lay.alt);
      le = (i % 2 == 0) ? launch_step_fused(c, dt, c->cap, a, b) : launch_step_fused(c, dt, c->cap, b, a);
    } else {
      le = launch_step_any(c, dt, c->cap);
    }
  }
  cudaGraph_t g = nullptr;
  e = cudaStreamEndCapture(c->cap, &g);
  if (le != cudaSuccess) { if (g) cudaGraphDestroy(g); return cuda_fail(le, "stage launch (capture)"); }
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
  e = cudaGraphInstantiate(&c->exec, g, 0);
  cudaGraphDestroy(g);
  if (e != cudaSuccess) { c->exec = nullptr; return cuda_fail(e, "cudaGraphInstantiate"); }
  c->graph_dt = dt;
  c->graph_variant = c->variant;
  return NLSE_OK;
}

__global__ void k_round_master(const double2* __restrict__ m, float2* __restrict__ o, int64_t total) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = m[i];
    o[i] = make_float2(float(v.x), float(v.y));
  }
}

// Wait for the stream, with *value (if given) the reduction's result: it lies beside the status word, one copy.
int read_status(nlse_ctx* c, double* value = nullptr) {
  unsigned char words[72];
  cudaError_t e = cudaMemcpyAsync(words, c->flag(), value ? 72 : 4, cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return cuda_fail(e, "status read");
  unsigned int flag = 0;
  memcpy(&flag, words, sizeof(flag));
  if (value) memcpy(value, words + 64, sizeof(double));
  if (flag & kFlagTimeoutBit) {
    // Report once and clear every status bit: nothing a timed-out step wrote
    // is valid (a non-finite value it produced included); the caller restores
    // Psi and the context stays usable.
    const unsigned int keep = 0;
    cudaMemcpyAsync(c->flag(), &keep, sizeof(keep), cudaMemcpyHostToDevice, c->stream);
    cudaStreamSynchronize(c->stream);
    return fail(NLSE_ETIMEOUT, "a bounded device-side wait gave up (a TMA copy did not complete)");
  }
  if (flag & 3u) return fail(NLSE_ENONFINITE, "non-finite value in Psi");
  return NLSE_OK;
}

}  // namespace

namespace nlse {
// Lets other translation units of the library report through nlse_last_error().
void record_last_error(const char* msg) { snprintf(g_err, sizeof(g_err), "%s", msg); }

// cuTensorMapEncodeTiled for other translation units (nullptr when unavailable).
void* tensor_map_encoder() { return reinterpret_cast<void*>(encode_fn()); }

__global__ void k_scale_v(const double* __restrict__ V, double s, int64_t n, double* __restrict__ Vs) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    Vs[i] = V[i] * s;
}

cudaError_t launch_scale_v(const double* V, double s, int64_t n, double* Vs, cudaStream_t stream) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  k_scale_v<<<(unsigned)b, 256, 0, stream>>>(V, s, n, Vs);
  return cudaGetLastError();
}

cudaError_t launch_round_master(const double2* master, float2* n32, int64_t total, cudaStream_t stream) {
  int64_t b = (total + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  k_round_master<<<(unsigned)b, 256, 0, stream>>>(master, n32, total);
  return cudaGetLastError();
}
}  // namespace nlse

extern "C" {

const char* nlse_last_error(void) { return g_err; }

size_t nlse_workspace_bytes(int dims, const int64_t* N, int dtype) {
  Layout L;
  if (!layout_for(dims, N, dtype, &L, nullptr)) return 0;
  return L.total;
}

double nlse_max_dt(int dims, double h, double a, int order, double vmax, double s_rho_max) {
  if (dims < 1 || dims > 3 || !(h > 0) || !(a > 0) || (order != 2 && order != 4)) return -1.0;
  // spectral radius of Lap on the grid: 4d/h^2 (CD), 16d/(3h^2) (2SHOC); RK4 reaches 2 sqrt(2) on i R
  const double rho = (order == 4 ? 16.0 * dims / 3.0 : 4.0 * dims) / (h * h);
  return 2.0 * sqrt(2.0) / (a * rho + fabs(vmax) + fabs(s_rho_max));
}

int nlse_create(nlse_t* out, int dims, const int64_t* N, double h, double a, double s, const void* V, int bc,
                int order, int dtype, void* psi, void* workspace, size_t ws_bytes, void* stream) {
  g_err[0] = 0;
  if (!out) return fail(NLSE_EINVAL, "out is NULL");
  *out = nullptr;
  Layout L;
  int64_t total = 0;
  if (!layout_for(dims, N, dtype, &L, &total))
    return fail(NLSE_EINVAL, "bad dims/N/dtype (dims in 1..3, every N >= 3, dtype 0..2)");
  if (!(h > 0) || !isfinite(h)) return fail(NLSE_EINVAL, "h must be > 0");
  if (!(a > 0) || !isfinite(a)) return fail(NLSE_EINVAL, "a must be > 0");
  if (!isfinite(s)) return fail(NLSE_EINVAL, "s must be finite");
  if (bc != NLSE_BC_DIRICHLET && bc != NLSE_BC_MSD && bc != NLSE_BC_L0 && bc != NLSE_BC_PERIODIC)
    return fail(NLSE_EINVAL, "bc must be 0, 1, 2 or 3");
  if (order != 2 && order != 4) return fail(NLSE_EINVAL, "order must be 2 or 4");
  if (!psi) return fail(NLSE_EINVAL, "psi is NULL");
  if (!workspace) return fail(NLSE_EINVAL, "workspace is NULL");
  if ((uintptr_t)workspace % kAlign) return fail(NLSE_EINVAL, "workspace must be 256-byte aligned");
  if ((uintptr_t)psi % 16 || (V && (uintptr_t)V % 8)) return fail(NLSE_EINVAL, "psi/V misaligned");
  if (ws_bytes < L.total) return fail(NLSE_ENOMEM, "workspace %zu bytes < %zu needed", ws_bytes, L.total);

  nlse_ctx* c = new nlse_ctx();
  memset(c, 0, sizeof(*c));
  c->d = dims;
  for (int k = 0; k < 3; ++k) c->n[k] = (k < dims) ? N[k] : 1;
  c->total = total;
  c->h = h; c->a = a; c->s = s;
  c->bc = bc; c->order = order; c->dtype = dtype;
  c->psi = psi; c->V = V;
  c->stream = (cudaStream_t)stream;
  c->ws = (char*)workspace;
  c->lay = L;
  // Default kernel per form and size, from timings of the paper's workloads (MSD, 2SHOC, us per step):
  // FP64 takes the exact-sum stencil on the tiled kernels, except where the grid is so small that a
  // step is bound by latency, not by the FP64 pipe's throughput, and the plain FP64 stencil's shorter
  // instruction chain wins: 3D grids of at most 2^15 sites (per-site kernels; 21^3: 21.8 against
  // 94.1 for the tiled exact-sum kernel, 32^3: 38.8 against 93.6; by time alone the line would lie higher, 46^3 74
  // against 85, 64^3 162 against 92, but moving it changes the arithmetic of the grids between) and 1D lines up to
  // 2^15 sites, several steps per launch where that is the faster form (lines_path; 2001 sites: 8.6 with MSD walls
  // against 19.2 for a launch per stage and 23.8 with the exact-sum stencil on a cluster; 32,000: 18.6 against 24.4
  // for the exact-sum stencil one thread per site; 49,000: 23.5 against 25.7).
  // FP64 planes take the exact-sum stencil where a whole step is one launch (step2x_fits) and above 80,000 sites
  // (316^2: 61.1 with the FP64 stencil, 54.0).  The planes between (274^2 to 282^2, and long or narrow ones) take the
  // FP64 stencil: where the operands' rounding is not taken back (Field::fine) its error is the smaller one (32 steps,
  // against 64 bits: 100x700 2.3e-16 and 3.0e-16, 5x6000 4.1e-16 and 9.2e-16).  Of its two forms the tiles (100x700
  // 48.7 against 53 for the exact-sum stencil then, 5x15000 43 against 51 for one thread per site), except on narrow
  // planes (12x5000: 86 with the tiles, 42 with one thread per site; 100x700 44).  A periodic plane of three or four
  // rows or columns is too narrow for the whole-step kernel's tiles (3x3 8.2 against 11.4, 3x4800 11.4 against 14.0
  // us with central differences).
  // The FP32 forms take the tiled kernel on 3D grids above 2^17 sites (64^3: 21.2 against 29.8 for one
  // thread per site, 128^3: 67.5 against 105; 40^3: 16.1 against 16.0).
  c->variant = (dtype == NLSE_C128) ? 2 : 1;
  if (dims == 3 && total <= (dtype == NLSE_C128 ? (int64_t(1) << 15) : (int64_t(1) << 17))) c->variant = 0;
  if (dims == 2 && dtype == NLSE_C128 && total <= 80000) {
    const int64_t side = N[0] < N[1] ? N[0] : N[1];
    if (!step2x_fits(int(N[0]), int(N[1]), bc == NLSE_BC_PERIODIC)) c->variant = side >= 8 && side <= 128 ? 0 : 1;
    else if (bc == NLSE_BC_PERIODIC && side < 5) c->variant = 1;
  }
  if (dims == 1 && dtype == NLSE_C128)
    c->variant = (total <= 2500 && line_ok(int(N[0]))) ? 1 : (total <= (int64_t(1) << 15) ? 0 : 3);
  c->tile_cfg = -1;
  c->spin_limit = kSpinLimit;
  c->graph_dt = -1.0;

  cudaError_t e = cudaMemsetAsync(c->at(L.status), 0, 256, c->stream);
  if (e == cudaSuccess && V) {
    e = launch_vmax(V, dtype == NLSE_C128, total, c->vbits(), c->stream);
    unsigned long long bits = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bits, c->vbits(), sizeof(bits), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    memcpy(&c->vmax, &bits, sizeof(double));
  }
  if (e == cudaSuccess && dims >= 2) {
    e = cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming);
    for (int i = 0; i < 2 && e == cudaSuccess && dims == 3; ++i) {
      e = cudaStreamCreateWithFlags(&c->side_yx[i], cudaStreamNonBlocking);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_join_yx[i], cudaEventDisableTiming);
    }
  }
  // Exact-sum stencil reference scale F0: the largest component of Psi0 below
  // 2^53 in fixed point.
  c->fixF = 52;
  if (e == cudaSuccess && dtype == NLSE_C128) {
    e = launch_vmax(psi, true, 2 * total, c->vbits(), c->stream);
    unsigned long long bits = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bits, c->vbits(), sizeof(bits), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    double pmax = 0.0;
    memcpy(&pmax, &bits, sizeof(double));
    if (pmax > 0.0 && isfinite(pmax)) {
      int ex = 0;
      frexp(pmax, &ex);              // pmax < 2^ex
      c->fixF = 56 - (ex + 3);
    }
  }
  if (e == cudaSuccess && dtype == NLSE_C128 && V) {   // V / cLF for the exact-sum stages
    const Field<P64> f = make_field<P64>(c, psi);
    e = launch_scale_v((const double*)V, 1.0 / f.cLF, total, (double*)c->at(L.vs), c->stream);
  }
  if (e == cudaSuccess && dtype == NLSE_C128) e = update_fix(c, psi, c->stream);
  if (e != cudaSuccess) {
    nlse_destroy(c);
    return cuda_fail(e, "nlse_create");
  }
  *out = c;
  return NLSE_OK;
}

int nlse_set_kernel(nlse_t c, int variant, int tile_cfg) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  if (variant < 0 || variant > 4) return fail(NLSE_EINVAL, "variant must be 0..4");
  if (tile_cfg < -1 || tile_cfg > 3) return fail(NLSE_EINVAL, "tile_cfg must be -1..3");
  c->variant = variant;
  c->tile_cfg = tile_cfg;
  c->chosen = true;
  drop_graph(c);
  return NLSE_OK;
}

int nlse_kernel_in_use(nlse_t c) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  if (fused_path(c)) return 4;
  if (line_path(c)) return 2;
  if (lines_path(c)) return c->variant == 0 ? 0 : 1;
  if (c->variant == 4) return c->d == 1 ? 0 : 1;
  if (c->d == 1) return (c->dtype == NLSE_C128 && c->variant >= 2) ? 3 : 0;
  if (c->dtype != NLSE_C128 && c->variant >= 2) return c->variant - 2;
  return c->variant;
}

int nlse_refresh_potential(nlse_t c) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  cudaError_t e = cudaSuccess;
  double vmax = 0.0;
  if (c->V) {
    e = launch_vmax(c->V, c->dtype == NLSE_C128, c->total, c->vbits(), c->stream);
    unsigned long long bits = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&bits, c->vbits(), sizeof(bits), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    memcpy(&vmax, &bits, sizeof(double));
    if (e == cudaSuccess && c->dtype == NLSE_C128) {
      const Field<P64> f = make_field<P64>(c, c->psi);
      e = launch_scale_v((const double*)c->V, 1.0 / f.cLF, c->total, (double*)c->at(c->lay.vs), c->stream);
    }
  }
  if (e != cudaSuccess) return cuda_fail(e, "nlse_refresh_potential");
  c->vmax = vmax;
  return NLSE_OK;
}

int nlse_step(nlse_t c, int64_t nsteps, double dt) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  if (nsteps < 0) return fail(NLSE_EINVAL, "nsteps < 0");
  if (!(dt > 0) || !isfinite(dt)) return fail(NLSE_EINVAL, "dt must be > 0");
  const double bound = nlse_max_dt(c->d, c->h, c->a, c->order, c->vmax, 0.0);
  if (dt > bound) return fail(NLSE_EUNSTABLE, "dt = %g above the RK4 linear stability bound %g", dt, bound);
  if (nsteps == 0) return NLSE_OK;
  cudaError_t e = cudaSuccess;
  if (c->dtype == NLSE_C64_ACC64 && !step2_path(c) && !lines_path(c))
    e = launch_round_master((const double2*)c->psi, (float2*)c->at(c->lay.pn32), c->total, c->stream);
  if (e != cudaSuccess) return cuda_fail(e, "round master");
  // the exact-sum scale of the state as the caller left it (stage 4 keeps it current from here on)
  if (step2x_path(c)) {
    e = cudaMemsetAsync(c->expo(), 0, 16, c->stream);
    if (e == cudaSuccess) e = launch_max_expo((const double*)c->psi, 2 * c->total, c->expo(), c->stream);
    if (e != cudaSuccess) return cuda_fail(e, "scale");
  } else if (c->exact() && (e = update_fix(c, c->psi, c->stream)) != cudaSuccess) return cuda_fail(e, "scale");
  if (line_path(c)) {   // 1D: the whole call on one thread-block cluster
    e = launch_line(c, nsteps, dt);
    if (e == cudaSuccess) return NLSE_OK;
    if (e != cudaErrorInvalidConfiguration) return cuda_fail(e, "line launch");
    cudaGetLastError();
    c->line_failed = true;   // cannot be co-scheduled here: the per-site kernel from now on
  }
  int64_t left = nsteps;
  if (nsteps >= kGraphSteps) {
    int rc = ensure_graph(c, dt);
    if (rc != NLSE_OK) return rc;
    for (; left >= kGraphSteps; left -= kGraphSteps) {
      e = cudaGraphLaunch(c->exec, c->stream);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
    }
  }
  if (lines_path(c) && left > 0) {   // launches of up to `per` steps; an odd number of them ends in the copy
    void *cur = c->psi, *nxt = step_alt(c);
    const int per = steps_per_launch(c);
    bool early = false;
    while (left > 0 && e == cudaSuccess) {
      const int k = left < per ? int(left) : per;
      e = launch_steps1_any(c, dt, k, c->stream, cur, nxt, early);
      early = true;
      void* t = cur;
      cur = nxt;
      nxt = t;
      left -= k;
    }
    if (e == cudaSuccess && cur != c->psi)
      e = cudaMemcpyAsync(c->psi, cur, (c->dtype == NLSE_C64 ? 8 : 16) * (size_t)c->total, cudaMemcpyDeviceToDevice,
                          c->stream);
    return e == cudaSuccess ? NLSE_OK : cuda_fail(e, "step launch");
  }
  if (step2_path(c) || step2x_path(c)) {   // pairs of steps end in Psi; an odd step goes through the copy and back
    void* alt = step_alt(c);
    for (int i = 0; left > 0 && e == cudaSuccess; left -= 2, i += 2) {
      e = launch_step2_any(c, dt, c->stream, c->psi, alt, i);
      if (e != cudaSuccess) break;
      if (left > 1) e = launch_step2_any(c, dt, c->stream, alt, c->psi, i + 1);
      else e = cudaMemcpyAsync(c->psi, alt, (c->dtype == NLSE_C64 ? 8 : 16) * (size_t)c->total,
                               cudaMemcpyDeviceToDevice, c->stream);
    }
    return e == cudaSuccess ? NLSE_OK : cuda_fail(e, "step launch");
  }
  for (; left > 0; --left) {
    e = launch_step_any(c, dt, c->stream);
    if (e != cudaSuccess) return cuda_fail(e, "stage launch");
  }
  return NLSE_OK;
}

int nlse_rhs(nlse_t c, const void* psi_in, void* F_out) {
  if (!c || !psi_in || !F_out) return fail(NLSE_EINVAL, "NULL argument");
  cudaError_t e;
  // A small plane whose whole step is one launch takes the exact sums for its steps alone (unless the caller chose
  // them): F by itself is the FP64 stencil, one launch instead of three (256^2 2SHOC 10.5 us, 27 with exact sums).
  const bool plain = !c->chosen && step2x_path(c);
  const bool exact = c->exact() && !plain;
  if (exact && (e = update_fix(c, psi_in, c->stream)) != cudaSuccess) return cuda_fail(e, "scale");
  auto run = [&](auto tag) {
    using T = decltype(tag);
    StageArgs<T> A;
    memset(&A, 0, sizeof(A));
    A.f = make_field<T>(c, psi_in);
    A.out = (typename T::C*)F_out;
    A.stage = 0;
    A.flag = c->flag();
    const bool g = std::is_same<T, P64>::value && exact;   // F in units of cLF: scale it back
    A.dtc = typename T::R(g ? A.f.cLF : 1.0);
    A.Vs = (g && c->V) ? (const typename T::VR*)c->at(c->lay.vs) : nullptr;
    return dispatch_stage<T>(c, A, nullptr, c->stream, plain ? 0 : -1);
  };
  if (c->dtype == NLSE_C128) e = run(P64{});
  else if (c->dtype == NLSE_C64) e = run(P32{});
  else e = run(PMix{});
  if (e != cudaSuccess) return cuda_fail(e, "rhs launch");
  return NLSE_OK;
}

int nlse_mass(nlse_t c, double* out_host) {
  if (!c || !out_host) return fail(NLSE_EINVAL, "NULL argument");
  cudaError_t e = launch_mass(c->psi, c->dtype != NLSE_C64, c->total, pow(c->h, c->d), c->partials(), c->result(),
                              c->flag(), c->done(), c->stream);
  double v = 0.0;
  if (e != cudaSuccess) return cuda_fail(e, "mass");
  int rc = read_status(c, &v);
  if (rc != NLSE_OK) return rc;
  *out_host = v;
  return NLSE_OK;
}

int nlse_energy(nlse_t c, double* out_host) {
  if (!c || !out_host) return fail(NLSE_EINVAL, "NULL argument");
  const double scale = pow(c->h, c->d);
  cudaError_t e;
  auto run = [&](auto tag) {
    using T = decltype(tag);
    Field<T> f = make_field<T>(c, c->psi);
    switch (c->d * 10 + c->order) {
      case 12: return launch_energy<T, 1, 2>(f, scale, c->partials(), c->result(), c->flag(), c->done(), c->stream);
      case 14: return launch_energy<T, 1, 4>(f, scale, c->partials(), c->result(), c->flag(), c->done(), c->stream);
      case 22: return launch_energy<T, 2, 2>(f, scale, c->partials(), c->result(), c->flag(), c->done(), c->stream);
      case 24: return launch_energy<T, 2, 4>(f, scale, c->partials(), c->result(), c->flag(), c->done(), c->stream);
      case 32: return launch_energy<T, 3, 2>(f, scale, c->partials(), c->result(), c->flag(), c->done(), c->stream);
      default: return launch_energy<T, 3, 4>(f, scale, c->partials(), c->result(), c->flag(), c->done(), c->stream);
    }
  };
  if (c->dtype == NLSE_C128) e = run(P64{});
  else if (c->dtype == NLSE_C64) e = run(E32{});
  else e = run(EMix{});
  double v = 0.0;
  if (e != cudaSuccess) return cuda_fail(e, "energy");
  int rc = read_status(c, &v);
  if (rc != NLSE_OK) return rc;
  *out_host = v;
  return NLSE_OK;
}

namespace {
std::mutex g_tune_mu;
std::map<std::string, int> g_tune;   // process-wide cache: context key -> tile_cfg

std::string tune_key(const nlse_ctx* c) {
  char b[160];
  snprintf(b, sizeof(b), "d%d n%lldx%lldx%lld t%d o%d bc%d v%d V%d", c->d, (long long)c->n[0], (long long)c->n[1],
           (long long)c->n[2], c->dtype, c->order, c->bc, c->variant, c->V ? 1 : 0);
  return b;
}

bool tune_file_lookup(const std::string& key, int* cfg) {
  const char* path = getenv("NLSE_TUNE_CACHE");
  if (!path) return false;
  FILE* f = fopen(path, "r");
  if (!f) return false;
  char line[256];
  bool found = false;
  while (fgets(line, sizeof(line), f)) {
    char* eq = strrchr(line, '=');
    if (!eq) continue;
    *eq = 0;
    if (key == line) { *cfg = atoi(eq + 1); found = true; }
  }
  fclose(f);
  return found;
}

void tune_file_store(const std::string& key, int cfg) {
  const char* path = getenv("NLSE_TUNE_CACHE");
  if (!path) return;
  FILE* f = fopen(path, "a");
  if (!f) return;
  fprintf(f, "%s=%d\n", key.c_str(), cfg);
  fclose(f);
}
}  // namespace

int nlse_autotune(nlse_t c, int* best_tile_cfg, float* best_ms) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  if (c->d == 1 || c->variant == 0 || c->variant == 3 || step2x_path(c)) {   // no tile to choose
    if (best_tile_cfg) *best_tile_cfg = -1;
    if (best_ms) *best_ms = 0.f;
    return NLSE_OK;
  }
  const std::string key = tune_key(c);
  int cfg = -1;
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) cfg = it->second;
  }
  float best = 0.f;
  if (cfg < 0 && tune_file_lookup(key, &cfg)) {
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune[key] = cfg;
  }
  if (cfg < 0) {
    // time stage 2 (the heaviest stage) for every tile; stage 1 fills its inputs.
    // Neither stage writes Psi.
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // the default where no launch of a step depends on the tile
    const bool same = columns_path(c) || (c->d == 2 && c->dtype != NLSE_C128 && !step2_path(c));
    const int saved = c->tile_cfg, only = same ? resolved_tile(c) : -1;
    best = 1e30f;
    cudaError_t e = cudaSuccess;
    if (c->dtype == NLSE_C64_ACC64)
      e = launch_round_master((const double2*)c->psi, (float2*)c->at(c->lay.pn32), c->total, c->stream);
    if (e == cudaSuccess && c->exact()) e = update_fix(c, c->psi, c->stream);
    for (int t = 0; t < 4 && e == cudaSuccess; ++t) {
      if (only >= 0 && t != only) continue;
      c->tile_cfg = t;
      const bool step2 = step2_path(c);   // one whole step, into Psi's ping-pong copy
      if (step2) e = launch_step2_any(c, 1e-12, c->stream, c->psi, step_alt(c), 0);
      else e = launch_stage_any(c, 1, 1e-12, c->stream);
      if (e == cudaSuccess && !step2) e = launch_stage_any(c, 2, 1e-12, c->stream);
      if (e == cudaSuccess) e = cudaEventRecord(e0, c->stream);
      for (int r = 0; r < 3 && e == cudaSuccess; ++r)
        e = step2 ? launch_step2_any(c, 1e-12, c->stream, c->psi, step_alt(c), 1) : launch_stage_any(c, 2, 1e-12, c->stream);
      if (e == cudaSuccess) e = cudaEventRecord(e1, c->stream);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e == cudaSuccess && ms / 3 < best) { best = ms / 3; cfg = t; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->tile_cfg = saved;
    if (e != cudaSuccess) return cuda_fail(e, "autotune");
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune[key] = cfg;
    tune_file_store(key, cfg);
  }
  c->tile_cfg = cfg;
  drop_graph(c);
  if (best_tile_cfg) *best_tile_cfg = cfg;
  if (best_ms) *best_ms = best;
  return NLSE_OK;
}

int nlse_debug_set(nlse_t c, int key, long long value) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  switch (key) {
    case NLSE_DEBUG_SPIN_LIMIT:
      if (value <= 0) return fail(NLSE_EINVAL, "spin limit must be > 0");
      c->spin_limit = value;
      break;
    case NLSE_DEBUG_EXTRA_TX:
      if (value < 0 || value > (1 << 20) || value % 16) return fail(NLSE_EINVAL, "extra_tx must be 0..2^20, multiple of 16");
      c->extra_tx = (unsigned int)value;
      break;
    case NLSE_DEBUG_FIX_OFFSET:
      if (value < -64 || value > 64) return fail(NLSE_EINVAL, "fix offset must be -64..64");
      c->fix_offset = (int)value;
      break;
    default:
      return fail(NLSE_EINVAL, "unknown debug key");
  }
  drop_graph(c);
  return NLSE_OK;
}

int nlse_sync(nlse_t c) {
  if (!c) return fail(NLSE_EINVAL, "NULL context");
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "pending error");
  return read_status(c);
}

int nlse_destroy(nlse_t c) {
  if (!c) return NLSE_OK;
  drop_graph(c);
  if (c->cap) cudaStreamDestroy(c->cap);
  for (int i = 0; i < 2; ++i) {
    if (c->side_yx[i]) cudaStreamDestroy(c->side_yx[i]);
    if (c->ev_join_yx[i]) cudaEventDestroy(c->ev_join_yx[i]);
  }
  if (c->side) cudaStreamDestroy(c->side);
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  if (c->ev_join) cudaEventDestroy(c->ev_join);
  delete c;
  return NLSE_OK;
}

}  // extern "C"
