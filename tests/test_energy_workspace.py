"""When the energy steps take the workspace of their stencil form: the decision against a fake of the CUDA calls (CPU)."""
import os
import shutil
import subprocess

import pytest

import paper_2609_21633_gb300 as tn
from paper_2609_21633_gb300 import build as tnbuild

CSRC = os.path.join(os.path.dirname(os.path.abspath(tn.__file__)), "csrc")

MAIN = r"""
#include <cassert>
#include <cstdio>
#include <set>
#include "energy_workspace.h"
// fake device: free memory, a failing allocation, a capturing stream
static size_t free_mem = 0;
static int fail_at = -1, allocs = 0;
static bool capturing = false;
static std::set<void*> live;
extern "C" {
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = free_mem, *t = 1000; return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  if (allocs++ == fail_at) return cudaErrorMemoryAllocation;
  *p = new char[n];
  live.insert(*p);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { assert(live.erase(p) == 1); delete[] (char*)p; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
}
int main() {
  {  // too little memory once, room later
    tn::RowsWorkspace w;
    free_mem = 399;
    if (tn::rows_ready(w, 80, 20, 0) || w.rows || !live.empty()) return 1;
    free_mem = 400;
    if (!tn::rows_ready(w, 80, 20, 0) || !w.rows || !w.wq || live.size() != 2) return 2;
    free_mem = 0;  // kept, whatever is free now
    const int n = allocs;
    if (!tn::rows_ready(w, 80, 20, 0) || allocs != n) return 3;
    cudaFree(w.rows), cudaFree(w.wq);
  }
  for (int at = 0; at < 2; ++at) {  // either allocation fails once
    tn::RowsWorkspace w;
    free_mem = 1000, allocs = 0, fail_at = at;
    if (tn::rows_ready(w, 80, 20, 0) || w.rows || w.wq || !live.empty()) return 4;
    fail_at = -1;
    if (!tn::rows_ready(w, 80, 20, 0) || live.size() != 2) return 5;
    cudaFree(w.rows), cudaFree(w.wq);
  }
  {  // a captured call allocates nothing and is no refusal for the next one
    tn::RowsWorkspace w;
    capturing = true, allocs = 0;
    if (tn::rows_ready(w, 80, 20, 0) || allocs) return 6;
    capturing = false;
    if (!tn::rows_ready(w, 80, 20, 0)) return 7;
    capturing = true;
    if (!tn::rows_ready(w, 80, 20, 0)) return 8;
  }
  return 0;
}
"""


def test_the_workspace_is_asked_for_again_after_a_refusal(tmp_path):
    inc = os.path.join(os.path.dirname(os.path.dirname(tnbuild.nvcc())), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-isystem", inc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
