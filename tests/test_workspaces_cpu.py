"""Workspaces of the products (Plan::grow): what a captured graph may point at
stays allocated while its tree stands.  Host code only, against a stand-in for
the CUDA allocator that counts."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "paper_2402_09531_gb300/csrc/dwfmm_internal.cuh"
#include <cstdio>
#include <set>
static std::set<void*> live;
static size_t room = 1 << 20;
extern "C" cudaError_t cudaMalloc(void** p, size_t n) {
  if (n > room) return cudaErrorMemoryAllocation;
  *p = malloc(n);
  live.insert(*p);
  return cudaSuccess;
}
extern "C" cudaError_t cudaFree(void* p) { live.erase(p); free(p); return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
static bool in_capture = false;
extern "C" cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = in_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
#define CHECK(c) if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; }
int main() {
  dw::Plan P;
  P.tree_gen = 5;
  P.grow(P.rot_pf, 100);
  float* narrow = P.rot_pf.p;
  P.grow(P.rot_pf, 80);
  CHECK(P.rot_pf.p == narrow && live.size() == 1)
  P.grow(P.rot_pf, 400);                       // a wider product of the same tree
  CHECK(P.rot_pf.p != narrow && live.count(narrow) && live.size() == 2)
  float* wide = P.rot_pf.p;
  room = 100;
  CHECK(!P.grow(P.rot_pf, 800))                // no room
  CHECK(P.rot_pf.p == wide && P.rot_pf.n == 400 && live.count(wide))
  room = 1 << 20;
  in_capture = true;
  CHECK(!P.grow(P.rot_pf, 800) && P.grow(P.rot_pf, 400) && P.rot_pf.p == wide && live.size() == 2)
  in_capture = false;
  P.outgrown.clear();                          // the tree goes
  ++P.tree_gen;
  CHECK(!live.count(narrow) && live.count(wide))
  P.grow(P.rot_pf, 300);                       // kept for the next one
  CHECK(P.rot_pf.p == wide && live.size() == 1)
  ++P.tree_gen;
  P.grow(P.rot_pf, 900);
  CHECK(live.size() == 1 && P.outgrown.empty())
  P.max_rhs = 16;
  CHECK(P.work_cols(1, 1, 99) == 1 && P.work_cols(2, 4, 99) == 4 && P.work_cols(5, 8, 6) == 6 && P.work_cols(5, 8, 5) == 5)
  P.max_rhs = 3;
  CHECK(P.work_cols(2, 4, 99) == 3 && P.work_cols(3, 4, 3) == 3)
  return 0;
}
"""


def test_workspaces_outlive_a_wider_product(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", ROOT, "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
