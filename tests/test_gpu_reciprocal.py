"""The reciprocal in the factor's chain of pivots, by itself, against CUDA's division and the exact quotient."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2602_04929_b200 import _build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "tb_rcp.cuh"
__global__ void k(const double* x, double* y, double* q, int n) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < n) {
    y[i] = tb::panel_rcp(x[i]);
    q[i] = 1.0 / x[i];
  }
}
extern "C" int reciprocals(const double* x, double* y, double* q, int n) {
  k<<<(n + 255) / 256, 256>>>(x, y, q, n);
  return cudaDeviceSynchronize();
}
"""


def test_reciprocal_of_a_pivot(tmp_path):
    """Half a unit of the last place from the last rounding and 2^-60 of the quotient from the iteration: 0.51 units."""
    import torch
    src, lib = tmp_path / "rcp.cu", tmp_path / "librcp.so"
    src.write_text(SOURCE)
    subprocess.run([_build._nvcc(), *_build.NVCC_FLAGS, "-shared", str(src), "-o", str(lib)], check=True, cwd=tmp_path)
    fn = ctypes.CDLL(str(lib)).reciprocals
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    g = np.random.default_rng(11)
    n = 1 << 20
    m = g.uniform(1.0, 2.0, n)
    m[:4096] = 1.0 + np.arange(4096) * 2.0 ** -52          # just above a power of two
    m[4096:8192] = 2.0 - np.arange(1, 4097) * 2.0 ** -52   # just below one
    e = np.where(g.random(n) < 0.5, g.integers(-54, 2, n), g.integers(-1000, 1000, n))  # pivots, and the whole range
    x = np.ldexp(m, e)
    t = torch.from_numpy(x).to("cuda:0")
    y, q = torch.empty_like(t), torch.empty_like(t)
    torch.cuda.synchronize()
    assert fn(t.data_ptr(), y.data_ptr(), q.data_ptr(), n) == 0
    y, q = y.cpu().numpy(), q.cpu().numpy()
    assert np.all(np.abs(y.view(np.int64) - q.view(np.int64)) <= 1)
    exact = 1.0 / x.astype(np.longdouble)                  # 64 bits
    ulp = np.spacing(q)
    assert float(np.max(np.abs(y.astype(np.longdouble) - exact) / ulp)) <= 0.511   # 0.51 and the 64 bits' own error
