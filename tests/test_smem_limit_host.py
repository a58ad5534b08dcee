"""The shared-memory opt-in is made once per device and tried again after a failure: smem_limit.h compiled with g++
against a stand-in for the two runtime calls it makes, and a source check that no other launch code keeps one."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1203_1263_gb300", "csrc")

STAND_IN = r"""
#pragma once
#include <cstddef>
enum cudaError_t { cudaSuccess = 0, cudaErrorUnknown = 999 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
extern int device, calls, bytes_seen;
extern cudaError_t set_result, get_result;
inline cudaError_t cudaGetDevice(int* d) { *d = device; return get_result; }
template <class K> cudaError_t cudaFuncSetAttribute(K, cudaFuncAttribute, int n) { ++calls; bytes_seen = n; return set_result; }
"""

PROGRAM = r"""
#include "smem_limit.h"
#include <cstdio>
int device = 0, calls = 0, bytes_seen = 0;
cudaError_t set_result = cudaSuccess, get_result = cudaSuccess;
static void kernel() {}
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
  nlse::SmemLimit a, b;
  CHECK(a.allow(kernel, 100000) == cudaSuccess && calls == 1 && bytes_seen == 100000);
  CHECK(a.allow(kernel, 100000) == cudaSuccess && calls == 1);       // once on this device
  device = 1;
  CHECK(a.allow(kernel, 100000) == cudaSuccess && calls == 2);       // and on the next
  CHECK(a.allow(kernel, 100000) == cudaSuccess && calls == 2);
  device = 0;
  CHECK(a.allow(kernel, 100000) == cudaSuccess && calls == 2);
  CHECK(b.allow(kernel, 5) == cudaSuccess && calls == 3);            // another kernel's own
  device = 63;
  set_result = cudaErrorUnknown;
  CHECK(a.allow(kernel, 1) == cudaErrorUnknown && calls == 4);       // a failure is reported and not kept
  set_result = cudaSuccess;
  CHECK(a.allow(kernel, 1) == cudaSuccess && calls == 5);
  CHECK(a.allow(kernel, 1) == cudaSuccess && calls == 5);
  device = 70;                                                       // beyond the mask: every time
  CHECK(a.allow(kernel, 1) == cudaSuccess && a.allow(kernel, 1) == cudaSuccess && calls == 7);
  get_result = cudaErrorUnknown;
  CHECK(a.allow(kernel, 1) == cudaErrorUnknown && calls == 7);
  return 0;
}
"""


def test_once_per_device_and_again_after_a_failure(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(STAND_IN)
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_launch_keeps_the_attribute_for_every_device():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        s = open(path).read()
        assert not re.search(r"static\s+const\s+cudaError_t", s), path
        for m in re.finditer(r"cudaFuncSetAttribute", s):   # direct calls: at every launch, or at every creation
            assert "static int per_sm" not in s[max(0, m.start() - 200):m.start()], path
