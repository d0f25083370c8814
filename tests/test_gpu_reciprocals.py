"""The iterated reciprocal and reciprocal square root of the kernels
(paper_2305_07181_gb300/csrc/phys.cuh), compiled into a program of their own:
over the float64 range in which argument and result are normal.  Bounds, in
units of 2^-53 of the result: the last rounding (1), and before it
  reciprocal   e^3 with e the estimate's error, 2^-20:                    < 1/16
  root         half the rounding of x r0 in e = 1 - x r0^2 (1/2), and the next
               term 5/16 e^3 with e = 2 2^-19 (0.16):                     < 0.7"""
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_07181_gb300", "csrc")

MAIN = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <vector>
#include "phys.cuh"
__global__ void eval(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = esplit::rcp64(x[i]);
  y[n + i] = esplit::rsqrt64(fabs(x[i]));
}
int main(int, char** v) {
  const int n = 1 << 18;
  std::vector<double> x(n), y(2 * n);
  FILE* f = std::fopen(v[1], "rb");
  if (!f || std::fread(x.data(), 8, n, f) != (size_t)n) return 2;
  std::fclose(f);
  double *dx, *dy;
  if (cudaMalloc(&dx, 8 * n) || cudaMalloc(&dy, 16 * n)) return 3;
  cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
  eval<<<n / 256, 256>>>(dx, dy, n);
  if (cudaMemcpy(y.data(), dy, 16 * n, cudaMemcpyDeviceToHost)) return 4;
  f = std::fopen(v[2], "wb");
  if (!f || std::fwrite(y.data(), 8, 2 * n, f) != 2 * (size_t)n) return 5;
  std::fclose(f);
  return 0;
}
"""


def test_reciprocals(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not torch.cuda.is_available() or not os.path.exists(nvcc):
        pytest.skip("no CUDA device or no nvcc")
    (tmp_path / "m.cu").write_text(MAIN)
    exe = str(tmp_path / "m")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(tmp_path / "m.cu"), "-o", exe], check=True)
    rng, n = np.random.default_rng(1), 1 << 18
    x = np.concatenate([rng.choice([-1.0, 1.0], n // 2) * 2.0 ** rng.uniform(-1020, 1020, n // 2),
                        rng.uniform(0.5, 4.0, n // 4), 1.0 + 2.0 ** -52 * rng.integers(-1000, 1000, n // 4)])
    x.tofile(tmp_path / "x")
    subprocess.run([exe, str(tmp_path / "x"), str(tmp_path / "y")], check=True)
    y = np.fromfile(tmp_path / "y")
    X = x.astype(np.longdouble)
    u = np.longdouble(2.0) ** -53
    assert np.all(np.abs(y[:n] * X - 1) <= u * (1 + 2.0 ** -4))
    # r = (1 + d)/sqrt(x): x r^2 - 1 = 2 d to first order
    r = y[n:].astype(np.longdouble)
    assert np.all(np.abs((np.abs(X) * r) * r - 1) <= 2 * u * 1.7 * (1 + 2.0 ** -40))
