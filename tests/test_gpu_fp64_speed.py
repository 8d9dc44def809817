"""The FP64 path's speed |u| (square root of a squared speed) at the edges of its range."""
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
  if ((int)threadIdx.x < n) y[threadIdx.x] = dg::fsqrt0(x[threadIdx.x]);
}
extern "C" int run(const double* x, double* y, int n) {
  k<<<1, 32>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_speed_of_zero_and_of_values_that_are_not_finite(tmp_path):
    """Zero gives zero, an ordinary value its root within 2 ulp, and a run that has blown up does not get a
    finite speed back."""
    import torch

    src, so = tmp_path / "f.cu", tmp_path / "f.so"
    src.write_text(SRC)
    cmd = [B._nvcc(), "-std=c++17", "-O3", "-shared", "-Xcompiler", "-fPIC", f"-I{B.INC}", f"-I{B.CSRC}"] + B.ARCH
    subprocess.run(cmd + ["-o", str(so), str(src)], check=True, capture_output=True)
    lib = ctypes.CDLL(os.fspath(so))
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    x = np.array([0.0, 1e-300, 2.0, 1e-280, 1e200, np.nan, np.inf])
    dx = torch.tensor(x, device="cuda")
    dy = torch.empty_like(dx)
    assert lib.run(dx.data_ptr(), dy.data_ptr(), len(x)) == 0
    y = dy.cpu().numpy()
    assert (y[:2] == 0.0).all()
    assert (np.abs(y[2:5] - np.sqrt(x[2:5])) <= 2 * np.spacing(np.sqrt(x[2:5]))).all()
    assert not np.isfinite(y[5:]).any()
