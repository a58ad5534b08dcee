"""The integer sums of wide_sum.cuh on the host: the header is compiled with g++ against a stand-in for the CUDA
runtime (the device intrinsics it names), and a block's accumulation is driven through its own add and merge."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_1263_gb300", "csrc")

STAND_IN = r"""
#pragma once
#include <cmath>
#include <cstring>
#include <cstdint>
#include <algorithm>
using std::max; using std::ldexp;
#define __device__
#define __forceinline__ inline
#define __shared__ static
struct Dim { int x; };
static Dim threadIdx = {0};
inline void __syncthreads() {}
inline int __reduce_max_sync(unsigned, int v) { return v; }
template <class T> inline T __shfl_down_sync(unsigned, T v, int) { return v; }
inline long long __double_as_longlong(double x) { long long r; std::memcpy(&r, &x, 8); return r; }
inline unsigned int __float_as_uint(float x) { unsigned int r; std::memcpy(&r, &x, 4); return r; }
inline int __clzll(long long x) { return x == 0 ? 64 : __builtin_clzll((unsigned long long)x); }
"""

# 2^k copies of a term by merging a sum with itself k times: pair (or value) must be 2^k times the term.
PROGRAM = r"""
#include "wide_sum.cuh"
#include <cstdio>
#include <cstdlib>
#include <limits>
int main(int, char** argv) {
  const int k = std::atoi(argv[1]);
  const double terms[] = {1.9999999999999998, -1.9999999999999998, 1.5 + std::ldexp(1.0, -52), 1e300, -3e-300};
  for (double x : terms) {
    nlse::WideSum w;
    w.add(x);
    for (int i = 0; i < k; ++i) w.merge(w);
    double s, c;
    w.pair(&s, &c);
    const double want = std::ldexp(x, k);
    if (!std::isfinite(want)) continue;
    if (s + c != want || (x > 0 && w.value() != want)) {
      std::printf("2^%d times %a: %a + %a, %a\n", k, x, s, c, w.value());
      return 1;
    }
  }
  // mixed magnitudes: 2^k of each, the smaller one far below the last bit of the larger
  nlse::WideSum a, b;
  a.add(1.75);
  b.add(std::ldexp(1.25, -60));
  a.merge(b);
  for (int i = 0; i < k; ++i) a.merge(a);
  double s, c;
  a.pair(&s, &c);
  if (s != std::ldexp(1.75, k) || c != std::ldexp(1.25, k - 60)) { std::printf("mixed: %a + %a\n", s, c); return 1; }
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide_sum")
    (d / "cuda_runtime.h").write_text(STAND_IN)
    (d / "main.cpp").write_text(PROGRAM)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(d), "-I", CSRC, str(d / "main.cpp"), "-o", exe], check=True)
    return exe


# 2^31 terms in one block: the most that a grid of 2^40 sites, the largest nlse_create accepts, gives one of 912 blocks
@pytest.mark.parametrize("k", [0, 1, 10, 20, 21, 22, 23, 26, 30, 31])
def test_a_block_of_full_terms_does_not_wrap(program, k):
    r = subprocess.run([program, str(k)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
