// Exact sums of many FP64 terms per thread on the integer pipe.
//
// GB300 issues FP64 at 1/64 of the FP32 rate, so a compensated FP64 sum (six
// FP64 instructions a term) bounds a reduction long before HBM does.  A term
// m 2^(e - 1075) (53-bit m) is instead added, shifted to a common exponent, to
// a 128-bit integer per thread: exact while the bits kept reach 2^42 below the
// last bit of the largest term seen, and otherwise off by less than 2^-94 of
// that term per addition.  A block's threads are combined as integers too; its
// total becomes an FP64 pair (sum, compensation) once.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace nlse {

struct WideSum {
  static constexpr int kGuard = 42;       // bits kept below the last bit of the largest term
  // Room: a term is below 2^(53 + 42) units, so up to 2^32 terms stay below 2^127.  A block of the 912 that a large
  // reduction has (kReduceBlocks) gets fewer than 2^31 of the 2^40 sites that a grid may have; the squares of FP32
  // components, two terms a site, are below 2^(48 + 42).
  unsigned long long lo = 0;
  long long hi = 0;                       // (hi:lo) in units of 2^(E - 1075 - kGuard)
  int E = 0;

  // rescale to exponent e >= E
  __device__ __forceinline__ void raise(int e) {
    const int d = e - E;
    if (d >= 127) { lo = 0; hi = 0; }
    else if (d >= 64) { lo = (unsigned long long)(hi >> (d - 64)); hi >>= 63; }
    else if (d > 0) { lo = (lo >> d) | ((unsigned long long)hi << (64 - d)); hi >>= d; }
    E = e;
  }
  __device__ __forceinline__ void merge(WideSum b) {
    const int e = max(E, b.E);
    raise(e);
    b.raise(e);
    const unsigned long long t = lo + b.lo;
    hi += b.hi + (t < lo ? 1 : 0);
    lo = t;
  }
  // add (negative ? -m : m) 2^(e - 1075), m < 2^53
  __device__ __forceinline__ void add(unsigned long long m, int e, bool negative) {
    if (e > E) raise(e);                  // rare: a larger exponent than any before
    const int s = kGuard - (E - e);       // left shift of m, <= kGuard
    unsigned long long l, h;
    if (s > 0) {
      l = m << s;
      h = m >> (64 - s);
    } else {
      l = s > -64 ? m >> -s : 0;
      h = 0;
    }
    if (negative) {
      l = 0ull - l;
      h = ~h + (l == 0ull ? 1ull : 0ull);
    }
    const unsigned long long t = lo + l;
    hi = (long long)((unsigned long long)hi + h + (t < lo ? 1ull : 0ull));
    lo = t;
  }
  // a finite FP64 term
  __device__ __forceinline__ void add(double x) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = int(u >> 52) & 0x7FF;
    add((u & 0x000FFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull), e ? e : 1, (u >> 63) != 0);
  }
  // x^2 of a finite FP32 value: its 24-bit mantissa squared, exactly
  __device__ __forceinline__ void add_square(float x) {
    const unsigned int u = __float_as_uint(x);
    const unsigned int e = (u >> 23) & 0xFFu;
    const unsigned int m = (u & 0x7FFFFFu) | (e ? 0x800000u : 0u);
    add((unsigned long long)m * m, 2 * (int(e ? e : 1) - 150) + 1075, false);
  }
  // a non-negative total, rounded: one conversion and one scaling (pair() is some forty dependent FP64 instructions)
  __device__ __forceinline__ double value() const {
    const unsigned long long h = (unsigned long long)hi;
    const int q = E - 1075 - kGuard;
    if (h == 0) return ldexp(double(lo), q);
    const int z = __clzll((long long)h), r = 64 - z;   // z >= 1
    const unsigned long long top = (h << z) | (lo >> r);
    return ldexp(double(top | ((lo << z) != 0 ? 1ull : 0ull)), q + r);   // 64 bits, the last one sticky
  }
  // the total as a rounded sum and what the rounding left
  __device__ __forceinline__ void pair(double* s, double* c) const {
    const bool neg = hi < 0;
    unsigned long long l = lo, h = (unsigned long long)hi;
    if (neg) {
      l = 0ull - l;
      h = ~h + (l == 0ull ? 1ull : 0ull);
    }
    // 128 bits in four 32-bit parts, each exact in FP64; the two upper first
    const int q = E - 1075 - kGuard;
    const double a = ldexp(double(h >> 32), q + 96), b = ldexp(double(h & 0xFFFFFFFFull), q + 64);
    const double d = ldexp(double(l >> 32), q + 32), f = ldexp(double(l & 0xFFFFFFFFull), q);
    const double t0 = a + b, r0 = b - (t0 - a);      // |a| >= |b| or a == 0: fast two-sum is exact
    const double t1 = t0 + d, r1 = d - (t1 - t0);
    const double t2 = t1 + f, r2 = f - (t2 - t1);
    const double r = r0 + (r1 + r2);
    *s = neg ? -t2 : t2;
    *c = neg ? -r : r;
  }
};

// The sum over a warp, in lane 0: one exponent for all first, so that a level is two shuffles and a 128-bit add (pairs
// rescaled at every level: 16 states of 64^2, two masses each, 4 us more).
__device__ __forceinline__ WideSum warp_wide_sum(WideSum v) {
  v.raise(__reduce_max_sync(0xffffffffu, v.E));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long l = __shfl_down_sync(0xffffffffu, v.lo, o);
    const long long h = __shfl_down_sync(0xffffffffu, v.hi, o);   // lanes past the end add values nobody reads
    const unsigned long long t = v.lo + l;
    v.hi = (long long)((unsigned long long)v.hi + (unsigned long long)h + (t < l ? 1ull : 0ull));
    v.lo = t;
  }
  return v;
}

// The sum over a block of THREADS threads, in thread 0.
template <int THREADS>
__device__ __forceinline__ WideSum block_wide_sum(WideSum v) {
  static_assert(THREADS <= 256 && THREADS % 32 == 0, "see kGuard");
  __shared__ long long sh[THREADS / 32];
  __shared__ unsigned long long sl[THREADS / 32];
  __shared__ int se[THREADS / 32];
  v = warp_wide_sum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sh[warp] = v.hi; sl[warp] = v.lo; se[warp] = v.E; }
  __syncthreads();
  if (warp == 0) {
    v = WideSum();
    if (lane < THREADS / 32) { v.hi = sh[lane]; v.lo = sl[lane]; v.E = se[lane]; }
    v = warp_wide_sum(v);
  }
  __syncthreads();   // the arrays may be used again
  return v;
}

}  // namespace nlse
