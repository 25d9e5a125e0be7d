"""The library's own exponentials, reciprocals and roots, compiled into a small
program and compared with the functions they stand for over their ranges."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import need_gpu  # noqa: E402
from paper_1110_1379_gb300 import build as B  # noqa: E402

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "frmg_kernels.cuh"
using namespace frmg;
template <int F>
__global__ void k_fun(const double *x, double *y, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double v = x[t];
  if (F == 0) y[t] = m_expm1_full((float)v);
  if (F == 1) y[t] = m_expm1_full2(make_float2(1.0f, (float)v)).y;
}
template <int F>
static int run(const double *x, double *y, long long n) {
  double *d = nullptr;
  if (cudaMalloc(&d, 2 * n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, x, n * sizeof(double), cudaMemcpyHostToDevice);
  k_fun<F><<<(unsigned)((n + 255) / 256), 256>>>(d, d + n, n);
  cudaMemcpy(y, d + n, n * sizeof(double), cudaMemcpyDeviceToHost);
  const int e = (int)cudaDeviceSynchronize();
  cudaFree(d);
  return e;
}
extern "C" int fun(int f, const double *x, double *y, long long n) {
  switch (f) {
    case 0: return run<0>(x, y, n);
    case 1: return run<1>(x, y, n);
  }
  return -1;
}
"""
NAMES = ["m_expm1_full", "m_expm1_full2"]


@pytest.fixture(scope="module")
def fun(tmp_path_factory):
    need_gpu()
    d = tmp_path_factory.mktemp("device_functions")
    src, lib = d / "fun.cu", d / "fun.so"
    src.write_text(SOURCE)
    subprocess.run([B.nvcc(), "-O3", "-std=c++17", *B.ARCH, "-Xcompiler", "-fPIC", "-shared",
                    "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), str(src), "-o",
                    str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).fun
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]

    def call(name, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        assert f(NAMES.index(name), x.ctypes.data, y.ctypes.data, x.size) == 0
        return y

    return call


@pytest.mark.parametrize("name", ["m_expm1_full", "m_expm1_full2"])
@pytest.mark.parametrize("lo,hi", [(-110.0, -80.0), (-80.0, -4.0), (-4.0, -0.3), (-0.4, 0.4),
                                   (0.3, 4.0), (4.0, 88.0)])
def test_fp32_expm1_of_the_full_variable(fun, name, lo, hi):
    """Its roundings (of the reduced argument, the series and the last sum) and
    the series' remainder add up to 1.6e-7 of the value."""
    x = np.linspace(lo, hi, 400001).astype(np.float32).astype(np.float64)
    ref = np.expm1(x)
    assert np.all(np.abs(fun(name, x) - ref) <= 1.6e-7 * np.abs(ref))


@pytest.mark.parametrize("name", ["m_expm1_full", "m_expm1_full2"])
def test_fp32_expm1_beyond_its_range(fun, name):
    far = np.array([-88.1, -89.0, -104.0, -1e3, -2e6, -1e7, -3e38, -np.inf])
    assert np.array_equal(fun(name, far), -np.ones(far.size))
    assert np.array_equal(fun(name, [88.8, 1e3, 2e6, 3e38, np.inf]), np.full(5, np.inf))
    assert np.all(np.isnan(fun(name, [np.nan])))
    assert np.array_equal(fun(name, [0.0, -0.0]), np.zeros(2))
