"""Device buffers whose allocation fails, on the host with a stand-in for cudaMalloc: the
buffer is empty afterwards, so that a later call sees that it has to be allocated."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SRC = r'''
#include <cstdio>
#include <cstdlib>
#include "amg_internal.cuh"
static bool room = true;
extern "C" cudaError_t cudaMalloc(void** p, size_t n) {
  if (!room) return cudaErrorMemoryAllocation;   // *p stays as it was
  *p = malloc(n);
  return cudaSuccess;
}
extern "C" cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
namespace amgp2 {
void check_cuda(cudaError_t e, const char* what, const char*, int) {
  if (e != cudaSuccess) throw Error{AMG_ERR_NOMEM, what};
}
}
int main() {
  amgp2::DBuf<double> b;
  b.alloc(10);
  room = false;
  try {
    b.alloc(20);
    return 1;
  } catch (const amgp2::Error& e) {
    if (e.code != AMG_ERR_NOMEM) return 2;
  }
  if (b.p || b.n || b.bytes()) return 3;
  room = true;
  b.alloc(20);
  return b.p && b.n == 20 ? 0 : 4;
}
'''


@pytest.mark.skipif(not shutil.which("g++") or not os.path.isdir(os.path.join(CUDA, "include")),
                    reason="needs g++ and the CUDA headers")
def test_failed_allocation_leaves_an_empty_buffer(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-w", "-I", os.path.join(CUDA, "include"), "-I",
                    os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1503_01287_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
