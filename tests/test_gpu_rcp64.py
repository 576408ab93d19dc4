"""rcp64 of csrc/series64.cuh against the correctly rounded FP64 quotient 1 / y:
at most one unit in the last place apart, over mantissas (random, next to one
and to two, around the approximate reciprocal's table steps) and over the
exponents its callers reach: sums of populations in units of 2^-62 of the
largest, 2^0 to 2^64, and differences of entropies, wide of both."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "series64.cuh"
__global__ void k(const double* y, double* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = elbm::rcp64(y[i]);
}
extern "C" int run(const double* y, double* r, int n) {
  double *a = nullptr, *b = nullptr;
  const size_t s = sizeof(double) * (size_t)n;
  cudaError_t e = cudaMalloc(&a, s);
  if (e == cudaSuccess) e = cudaMalloc(&b, s);
  if (e == cudaSuccess) e = cudaMemcpy(a, y, s, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k<<<(n + 255) / 256, 256>>>(a, b, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(r, b, s, cudaMemcpyDeviceToHost);
  cudaFree(a);
  cudaFree(b);
  return (int)e;
}
"""


def test_rcp64(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1904_00866_gb300 import _build
    src, lib = tmp_path / "rcp.cu", tmp_path / "librcp.so"
    src.write_text(SOURCE)
    subprocess.run([_build.nvcc()] + _build.ARCH + _build.FLAGS +
                   ["-I", _build.CSRC, "-Xcompiler", "-fvisibility=default",
                    "-shared", "-o", str(lib), str(src)], check=True)
    run = ctypes.CDLL(str(lib)).run
    rng = np.random.default_rng(1)
    n = 1 << 20
    m = 1 + rng.integers(0, 1 << 52, n) * 2.0 ** -52
    m[: n // 4] = 1 + (np.arange(n // 4) % 8192) / 8192 + rng.integers(
        -3, 4, n // 4) * 2.0 ** -52
    m[0:64] = 1 + np.arange(64) * 2.0 ** -52
    m[64:128] = 2 - (1 + np.arange(64)) * 2.0 ** -52
    e = rng.integers(-900, 900, n)
    e[: n // 2] = rng.integers(0, 65, n // 2)
    y = np.ldexp(np.abs(m), e)
    r = np.empty_like(y)
    dp = ctypes.POINTER(ctypes.c_double)
    assert run(y.ctypes.data_as(dp), r.ctypes.data_as(dp), n) == 0
    ulp = np.abs(r.view(np.int64) - (1.0 / y).view(np.int64))
    assert ulp.max() <= 1, (ulp.max(), y[ulp.argmax()])
