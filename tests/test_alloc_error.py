"""A cudaMalloc that fails leaves no error behind.  The runtime keeps a failed call's error until it is
asked for, and the launches check for one, so a caller that takes SLDM_ENOMEM and goes another way (the
Schur inverse in FP64, the far field with a smaller workspace) would fail at its next launch.  DBuf is
compiled here against a runtime of a few lines whose cudaMalloc fails."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06184_gb300", "csrc")

SRC = r"""
#include "internal.h"
static cudaError_t last = cudaSuccess;
extern "C" {
cudaError_t cudaMalloc(void**, size_t) { return last = cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
}
namespace sldm {
static size_t held = 0;
void budget_take(size_t b) { held += b; }
void budget_give(size_t b) { held -= b; }
}
int main() {
  sldm::DBuf<double> b;
  int code = 0;
  try {
    b.alloc(100);
  } catch (const sldm::Error& e) {
    code = e.code;
  }
  if (code != SLDM_ENOMEM || b.p || b.n || sldm::held) return 1;
  return cudaGetLastError() == cudaSuccess ? 0 : 2;  // what the next launch's check sees
}
"""


def test_failed_allocation_leaves_no_runtime_error(tmp_path):
    (tmp_path / "a.cpp").write_text(SRC)
    exe = str(tmp_path / "a")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", str(tmp_path / "a.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
