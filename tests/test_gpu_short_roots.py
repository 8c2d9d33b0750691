"""The short reciprocal square root and reciprocal of the factorisations, against exact arithmetic.  The relative error
is bounded by that of the series cut after the second power of e and that of the roundings: rsqrt_fast 2.5 delta^3 +
1.5 2^-53 (e is rounded at 2^-53 and enters halved, the last operation rounds once), rcp_fast delta^3 + 2^-53, where
delta, the relative error of the hardware's start value, is measured here too and assumed to be at most 2^-19."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include "gcamps_roots.cuh"
__global__ void k(const double* a, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double r, q;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a[i]));
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(q) : "d"(a[i]));
  out[i] = gcx::rsqrt_fast(a[i]);
  out[n + i] = gcx::rcp_fast(a[i]);
  out[2 * n + i] = r;
  out[3 * n + i] = q;
}
extern "C" int roots(const double* a, double* out, int n) {
  double *da = nullptr, *dout = nullptr;
  cudaError_t e = cudaMalloc(&da, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&dout, 4 * n * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(da, a, n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k<<<(n + 255) / 256, 256>>>(da, dout, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, dout, 4 * n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(da);
  cudaFree(dout);
  return (int)e;
}
"""

DELTA, U = Fraction(1, 2 ** 19), Fraction(1, 2 ** 53)


def _inputs():
    """The exponents the callers pass (squares of norms down to 1e-290, the guards' 2^+-900) and every mantissa edge."""
    rng = np.random.default_rng(7)
    wide = np.ldexp(1.0 + rng.random(40000), rng.integers(-962, 900, 40000))
    near = 1.0 + 3.0 * rng.random(40000)
    edges = np.array([m * 2.0 ** e for e in (-963, -962, -901, -900, -899, -2, -1, 0, 1, 2, 899, 900)
                      for m in (1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -20, 1.5, 2.0 - 2.0 ** -20, 2.0 - 2.0 ** -52)])
    return np.concatenate([wide, near, edges])


def test_roots_within_their_bounds(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300 import build
    src, lib = tmp_path / "roots.cu", tmp_path / "roots.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-O3", "-I", build.CSRC, "-shared", "-Xcompiler", "-fPIC",
                    "-o", str(lib), str(src)], check=True, timeout=300)
    a = np.ascontiguousarray(_inputs())
    out = np.zeros((4, len(a)))
    f = ctypes.CDLL(os.fspath(lib)).roots
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    assert f(a.ctypes.data, out.ctypes.data, len(a)) == 0
    worst = [Fraction(0)] * 4
    for i in range(len(a)):
        x = Fraction(a[i])
        # y = (1 + t) / sqrt(x): x y^2 - 1 = 2 t + t^2; |t| <= |x y^2 - 1| / 2 (1 + |x y^2 - 1|)
        for row, square in ((0, True), (1, False), (2, True), (3, False)):
            y = Fraction(out[row, i])
            e = abs(x * y * y - 1) if square else abs(x * y - 1)
            t = e / 2 * (1 + e) if square else e
            if t > worst[row]:
                worst[row] = t
    print("units of 2^-53:", [float(w / U) for w in worst])
    assert worst[2] <= DELTA and worst[3] <= DELTA
    # the products of small terms (e^2 2^-53 and the like) are covered by the last factor
    assert worst[0] <= (Fraction(5, 2) * DELTA ** 3 + Fraction(3, 2) * U) * (1 + 4 * DELTA)
    assert worst[1] <= (DELTA ** 3 + U) * (1 + 4 * DELTA)
