"""The kernels' own pair sums (pair32.cuh) against FP64: (h + l) v over a list of terms, then times a pair, as the
charge rows take it.

Of n terms with P = sum |terms|: the second number takes two errors of at most 2^-24 P per term, exactly, and
rounds after each, so it is at most 2 k 2^-24 P after k terms and its roundings add up to 2 n (n + 1)
2^-48 P; 2^-147 n absolute where the terms are too small for their errors to be FP32 numbers.  Infinities and
NaN as FP64 gives them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06184_gb300", "csrc")
SRC = r"""
#include "pair32.cuh"
using namespace sldm;
__global__ void fn(int n, int m, const double* x, const float* v, double s, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  P32 a;
  for (int k = 0; k < m; ++k) {
    const double c = x[i * m + k];
    const float h = float(c);
    a.fma(h, float(c - double(h)), v[i * m + k]);
  }
  a.get(out[i]);
  const float h = float(s);
  a.scaled(h, float(s - double(h))).get(out[n + i]);
  float f;
  a.get(f);
  out[2 * n + i] = f;
}
extern "C" int run(int n, int m, const double* x, const float* v, double s, double* out) {
  fn<<<(n + 127) / 128, 128>>>(n, m, x, v, s, out);
  return int(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import torch
    from paper_2106_06184_gb300 import build
    d = tmp_path_factory.mktemp("p32")
    (d / "p.cu").write_text(SRC)
    so = str(d / "p.so")
    subprocess.run([build._nvcc(), "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", *build.ARCH, "-I", CSRC, str(d / "p.cu"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)

    def f(x, v, s):
        n, m = x.shape
        dx, dv = torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda()
        out = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        p = [ctypes.c_void_p(t.data_ptr()) for t in (dx, dv, out)]
        assert lib.run(n, m, p[0], p[1], ctypes.c_double(s), p[2]) == 0
        return out.cpu().numpy()
    return f


@pytest.mark.parametrize("scale", [1.0, 1e30, 1e-20, 1e-32, 1e-38])
def test_sums(call, scale):
    rng = np.random.default_rng(8)
    x = rng.standard_normal((4000, 12)) * 10.0 ** rng.uniform(-3, 3, (4000, 12))
    v = (rng.standard_normal((4000, 12)) * scale).astype(np.float32)
    x[:100, 1:], v[:100, 1:] = -x[:100, :1], v[:100, :1]  # cancellation
    s = 0.37
    got = call(x, v, s)
    t = x.astype(np.longdouble) * v.astype(np.longdouble)
    ref, lim = t.sum(1), 2 * 12 * 13 * 2.0 ** -48 * np.abs(t).sum(1) + 2.0 ** -147 * 12
    assert np.all(np.abs(got[0] - ref) <= lim)
    assert np.all(np.abs(got[1] - s * ref) <= lim)
    assert np.all(np.abs(got[2] - ref) <= lim + 2.0 ** -24 * np.abs(ref) + 2.0 ** -149)


def test_infinities_and_nan(call):
    inf, big = np.inf, 3e38
    v = np.array([[1, inf, 2], [-inf, 1, 1], [inf, -inf, 1], [np.nan, 1, 1], [big, big, 1], [-big, -big, 1]], np.float32)
    got = call(np.ones_like(v, dtype=np.float64), v, 0.5)
    for row in got[:2]:
        assert row[0] == inf and row[1] == -inf and np.isnan(row[2]) and np.isnan(row[3])
        assert row[4] == inf and row[5] == -inf  # beyond FP32's range
