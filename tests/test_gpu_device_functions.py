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
  if (F == 2) y[t] = f64_expm1(v);
  if (F == 3) y[t] = f64_exp(v);
  if (F == 4) y[t] = f64_rcp(v);
  if (F == 5) y[t] = f64_rsqrt(v);
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
    case 2: return run<2>(x, y, n);
    case 3: return run<3>(x, y, n);
    case 4: return run<4>(x, y, n);
    case 5: return run<5>(x, y, n);
  }
  return -1;
}
"""
NAMES = ["m_expm1_full", "m_expm1_full2", "f64_expm1", "f64_exp", "f64_rcp", "f64_rsqrt"]


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


def _ulps(y, ref):
    """Distance of FP64 values from extended-precision ones, in units of the last
    FP64 place of the latter."""
    return np.abs((y.astype(np.longdouble) - ref)
                  / np.spacing(np.abs(ref).astype(np.float64))).astype(np.float64).max()


LN2_32 = np.log(2.0) / 32


@pytest.mark.parametrize("sign", [-1.0, 1.0])
@pytest.mark.parametrize("lo,hi,bound", [(1e-12, LN2_32, 1.0), (LN2_32, 0.035, 2.5),
                                         (0.035, 0.1, 1.5), (0.1, 0.75, 1.25), (0.7, 40.0, 1.25),
                                         (40.0, 699.9, 1.25)])
def test_fp64_exponentials(fun, sign, lo, hi, bound):
    """All sixteen entries of the table (steps of ln2 / 16 = 0.043), both signs.
    expm1: half an ulp per rounding of a term of the result's size (the result
    itself; r, r + dt and p where they are as large as it), and what the terms
    below them add."""
    rng = np.random.default_rng(3)
    x = sign * np.concatenate([np.linspace(lo, hi, 50001), rng.uniform(lo, hi, 50001)])
    xl = x.astype(np.longdouble)
    assert _ulps(fun("f64_expm1", x), np.expm1(xl)) <= bound
    assert _ulps(fun("f64_exp", x), np.exp(xl)) <= 0.6


def test_fp64_exponentials_beyond_their_range(fun):
    """What the library's functions give (subnormals within an ulp)."""
    x = np.array([700.0, 705.3, 709.7, 709.8, 1e4, np.inf, -700.0, -709.0, -720.5, -744.0, -746.0,
                  -1e4, -np.inf, 0.0])
    with np.errstate(over="ignore", under="ignore"):
        e, m = np.exp(x), np.expm1(x)
    for name, ref in (("f64_exp", e), ("f64_expm1", m)):
        y = fun(name, x)
        fin = np.isfinite(ref)
        assert np.array_equal(y[~fin], ref[~fin])
        assert np.all(np.abs(y[fin] - ref[fin]) <= 2 * np.spacing(np.abs(ref[fin])))
        assert np.isnan(fun(name, [np.nan])[0])


@pytest.mark.parametrize("name,bound", [("f64_rcp", 0.55), ("f64_rsqrt", 1.05)])
def test_fp64_reciprocal_and_root(fun, name, bound):
    """Significands over two binades (the root's period), exponents over the range
    they are used on."""
    rng = np.random.default_rng(4)
    m = np.concatenate([np.linspace(1.0, 4.0, 100001), rng.uniform(1.0, 4.0, 100001),
                        np.nextafter([1.0, 2.0, 4.0], 0.0), np.nextafter([1.0, 2.0], 4.0)])
    for e in (-1001, -500, -3, 0, 1, 499, 980):
        x = np.ldexp(m, e)
        xl = x.astype(np.longdouble)
        ref = 1 / xl if name == "f64_rcp" else 1 / np.sqrt(xl)
        assert _ulps(fun(name, x), ref) <= bound
        if name == "f64_rcp":
            assert _ulps(fun(name, -x), -ref) <= bound
