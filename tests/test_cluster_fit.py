"""Whether a device schedules a kernel's clusters is asked for once, at the most shared memory that a launch of
it may take.  Compiled here against a runtime of a few lines: a device that holds a cluster of
16 CTAs only while each takes 64 KB or less must say no, whatever is launched first, and one that holds
them at the limit yes, without a second question."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06184_gb300", "csrc")

SRC = r"""
#include "cluster.h"
static size_t holds, set = 0;
static int asked = 0, cleared = 0;
extern "C" {
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) set = size_t(v);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  ++asked;
  *n = c->attrs[0].val.clusterDim.x == 16 && c->dynamicSmemBytes <= set && c->dynamicSmemBytes <= holds ? 3 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { ++cleared; return cudaSuccess; }
}
int main(int argc, char**) {
  holds = size_t(argc > 1 ? 64 : 128) * 1024;
  sldm::ClusterFit f;
  const bool want = argc == 1;
  for (int i = 0; i < 3; ++i)
    if (sldm::cluster_fits(f, 0, nullptr, 16, 512, 128 * 1024) != want) return 1;
  return asked == 1 && set == 128 * 1024 ? 0 : 2;
}
"""


@pytest.mark.parametrize("args", [[], ["small"]])
def test_asked_at_the_limit(tmp_path, args):
    (tmp_path / "a.cpp").write_text(SRC)
    exe = str(tmp_path / "a")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", str(tmp_path / "a.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe, *args]).returncode == 0


def test_steps_are_refused_above_the_limit_they_were_asked_at():
    """Both callers pass one constant to the question and hold their launches to it."""
    src = open(os.path.join(CSRC, "gmres_dev.cu")).read()
    assert "smem > GS_SMEM_MAX || !cluster_fits(" in src and "GS_THREADS, GS_SMEM_MAX)" in src
    src = open(os.path.join(CSRC, "lu_blocked.cu")).read()
    assert "if (smem > LIMIT) return false;" in src and "PC_THREADS, LIMIT)" in src
