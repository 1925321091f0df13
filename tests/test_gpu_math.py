"""The functions of one argument that the fills evaluate by tables and series instead of CUDA's (fill_dev.cuh, widen.cuh), over
the ranges they are used on, against long double (at least 64 bits) and, where it is exact, the conversion itself.

Bounds, from the operations: wave_cis one table entry (CUDA's sincospi: 1 ulp below 1, 1.1e-16), two
roundings of 0.56e-16, series 1e-17: 2.5e-16 absolute whatever the phase.  wave_exp2 the same relative to
1: entry 2.2e-16, rounding 1.1e-16, series 4e-17: 4e-16.  rsqrt_pos and recip_pos: the hardware's
2^-20 cubed, the residual's rounding (0.6e-16, halved or none) and the last one, 1.1e-16: 2.3e-16 and
1.7e-16 (CUDA's rsqrt and quotient: 2.2e-16 and 1.1e-16).  log2_pos: entry 1.1e-16, two roundings of the sum."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_06184_gb300", "csrc")
SRC = r"""
#include "internal.h"
#include "fill_dev.cuh"
#include "widen.cuh"
using namespace sldm;
__global__ void fn(int which, int n, const double* x, double* a, double* b) {
  __shared__ WaveTab T;
  __shared__ LogTab L;
  wave_tab_fill(T, true);
  log_tab_fill(L);
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (which == 0) wave_cis(T, x[i], a[i], b[i]);
  if (which == 1) a[i] = wave_exp2(T, x[i]);
  if (which == 2) a[i] = rsqrt_pos(x[i]);
  if (which == 3) a[i] = recip_pos(x[i]);
  if (which == 4) a[i] = log2_pos(L, x[i]);
  if (which == 5) a[i] = widen(__int_as_float(int(unsigned(x[i]))));
}
extern "C" int run(int which, int n, const double* x, double* a, double* b) {
  fn<<<(n + 255) / 256, 256>>>(which, n, x, a, b);
  return int(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import torch
    from paper_2106_06184_gb300 import build
    d = tmp_path_factory.mktemp("fn")
    (d / "fn.cu").write_text(SRC)
    so = str(d / "fn.so")
    subprocess.run([build._nvcc(), "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", *build.ARCH, "-I", CSRC,
                    str(d / "fn.cu"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def f(which, x):
        x = torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()
        a, b = torch.zeros_like(x), torch.zeros_like(x)
        p = [ctypes.c_void_p(t.data_ptr()) for t in (x, a, b)]
        assert lib.run(which, len(x), *p) == 0
        return a.cpu().numpy(), b.cpu().numpy()
    return f


def wide(n, lo, hi, rng):
    return np.exp(rng.uniform(np.log(lo), np.log(hi), n))


def test_wave_cis(call):
    rng = np.random.default_rng(1)
    y = np.concatenate([[0.0, 0.5, -0.5, 1.5, 127.5, 128.0, 1e-300, 2.0 ** 50 + 1], np.arange(-600, 600) / 2,
                        *[s * wide(4000, a, b, rng) for s in (1, -1) for a, b in ((1e-9, 1.0), (1.0, 2.0 ** 20), (2.0 ** 20, 2.0 ** 45))]])
    c, s = call(0, y)
    a = np.fmod(y, 256.0).astype(np.longdouble) * (2 * np.arccos(np.longdouble(-1)) / 256)
    assert np.max(np.abs(c - np.cos(a))) <= 2.5e-16 and np.max(np.abs(s - np.sin(a))) <= 2.5e-16


def test_wave_exp2(call):
    rng = np.random.default_rng(2)
    lim = 1021 * 256.0
    y = np.concatenate([rng.uniform(-lim, lim, 20000), rng.uniform(-2, 2, 4000), [0.0, 0.5, -0.5, -lim + 0.25, lim - 0.25]])
    e, _ = call(1, y)
    ref = np.exp2(y.astype(np.longdouble) / 256)
    assert np.max(np.abs(e / ref - 1)) <= 4e-16
    e, _ = call(1, np.array([-lim, -1e6, -1e300, -np.inf]))
    assert np.all(e == 0.0)  # below 2^-1021
    e, _ = call(1, np.array([lim, 1e6, 1e300, np.inf]))
    assert np.all(np.isinf(e) & (e > 0))


def test_roots_and_reciprocals(call):
    rng = np.random.default_rng(3)
    x = np.concatenate([wide(20000, 1e-300, 1e300, rng), wide(4000, 0.25, 4.0, rng), [1.0, 2.0, 4.0, 2.0 ** -1000, 2.0 ** 1000]])
    r, _ = call(2, x)
    assert np.max(np.abs(r * np.sqrt(x.astype(np.longdouble)) - 1)) <= 2.3e-16
    r, _ = call(3, x)
    assert np.max(np.abs(r * x.astype(np.longdouble) - 1)) <= 1.7e-16


def test_log2(call):
    rng = np.random.default_rng(4)
    x = np.concatenate([wide(20000, 1e-300, 1e300, rng), wide(8000, 0.5, 2.0, rng), 1 + np.arange(-9, 10) * 2.0 ** -52, 2.0 ** np.arange(-900, 900)])
    v, _ = call(4, x)
    ref = np.log2(x.astype(np.longdouble))
    assert np.all(np.abs(v - ref) <= 1.3e-16 + 2.3e-16 * np.abs(ref))


def test_widen_is_the_conversion(call):
    """Every class of FP32 number: zeros, denormals, normals, infinities, NaN."""
    rng = np.random.default_rng(5)
    bits = np.concatenate([rng.integers(0, 2 ** 32, 20000), rng.integers(0, 2 ** 23, 4000), 2 ** 31 + rng.integers(0, 2 ** 23, 4000),
                           [0, 1, 2 ** 31, 2 ** 31 + 1, 0x007fffff, 0x00800000, 0x7f7fffff, 0x7f800000, 0xff800000, 0x7f800001, 0x7fc00000]])
    v, _ = call(5, bits.astype(np.float64))
    with np.errstate(invalid="ignore"):
        ref = bits.astype(np.uint32).view(np.float32).astype(np.float64)
    nan = np.isnan(ref)
    assert np.all(np.isnan(v[nan])) and np.array_equal(v[~nan].view(np.uint64), ref[~nan].view(np.uint64))
