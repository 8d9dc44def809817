"""The FP64 path's reciprocal, inverse square root and inverse cube root (one Householder step from a
20-bit seed) against extended precision, over the exponents that depths, speeds and lengths take."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2307_14302_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = """
#include "stage.cuh"
__global__ void k(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double inv, f;
  dg::depth_inverse(x[i], 0, inv, f);
  y[i] = dg::hh_rcp(x[i]);
  y[n + i] = dg::hh_rsqrt(x[i]);
  y[2 * n + i] = dg::hh_rcbrt(x[i]);
  y[3 * n + i] = inv;
  y[4 * n + i] = f;
}
extern "C" int run(const double* x, double* y, int n) {
  k<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_ulp_errors(tmp_path):
    """Bounds from the operation counts: a final rounding (half an ulp) plus the rounding of the
    residual's products, scaled by 1/k: 1, 2, 2 ulp; 1/H corrected once: 1 ulp; H^(-4/3): one more product
    and the cube root's own 2."""
    import torch

    src, so = tmp_path / "f.cu", tmp_path / "f.so"
    src.write_text(SRC)
    cmd = [B._nvcc(), "-std=c++17", "-O3", "-shared", "-Xcompiler", "-fPIC", f"-I{B.INC}", f"-I{B.CSRC}"] + B.ARCH
    subprocess.run(cmd + ["-o", str(so), str(src)], check=True, capture_output=True)
    lib = ctypes.CDLL(os.fspath(so))
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    rng = np.random.default_rng(8)
    n = 1_000_000
    x = np.concatenate([2.0 ** rng.uniform(-60, 60, n - 3000), np.linspace(1, 8, 2000), 2.0 ** np.arange(-500.0, 500.0)])
    dx = torch.tensor(x, device="cuda")
    dy = torch.empty((5, n), dtype=torch.float64, device="cuda")
    assert lib.run(dx.data_ptr(), dy.data_ptr(), n) == 0
    y = dy.cpu().numpy()
    q = x.astype(np.longdouble)
    c = np.cbrt(q)
    c = c - (c * c * c - q) / (3 * c * c)
    want = [1 / q, 1 / np.sqrt(q), 1 / c, 1 / q, 1 / (q * c)]
    for got, w, bound in zip(y, want, (1.0, 2.0, 2.0, 1.0, 3.5)):
        ulp = np.spacing(np.abs(w.astype(np.float64))).astype(np.longdouble)
        assert float((np.abs(got - w) / ulp).max()) <= bound
