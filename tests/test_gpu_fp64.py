"""The FP64 functions of csrc/fp64.cuh (reciprocal, square roots, exponential,
half-range error function), which keep seeds, range reduction and exponents on the
integer and FP32 units, against values in 50 digits.

Bounds, in units of the last place of the result: a Newton step from a seed good to
2^-45 leaves the rounding of its last FMA (rcp, sqrt: 0.5, plus the terms it drops:
0.51); rsqrt adds the rounding of x y (1); exp adds the rounding of its table entry
(0.5) and of its argument's reduction (1.1); erfc/2 is a polynomial whose argument
d = x - k/32 is exact, so the roundings of its last two operations count (1.1). Arguments outside the fast range must give the library's value.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2304_09485_gb300 import _native

pytestmark = pytest.mark.gpu

SRC = r"""
#include "fp64.cuh"
using namespace hgks;
__global__ void k(int f, int n, const double *x, double *y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  y[i] = f == 0 ? rcp(v) : f == 1 ? rsqrt64(v) : f == 2 ? sqrt64(v) : f == 3 ? exp64(v) : f == 4 ? half_erfc64(v)
       : f == 5 ? (positive(v) ? 1.0 : 0.0) : min_positive(v, 1.0);
}
extern "C" int run(int f, int n, const double *x, double *y) {
  double *d;
  if (cudaMalloc(&d, 2 * sizeof(double) * n)) return 1;
  cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(f, n, d, d + n);
  const int rc = cudaMemcpy(y, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(d);
  return rc;
}
"""


@pytest.fixture(scope="module")
def run(cuda, tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64")
    src, so = str(d / "fp64.cu"), str(d / "libfp64.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([_native._nvcc(), *_native.ARCH, "-O3", "-std=c++17", "-I", _native.CSRC, "-shared", "-Xcompiler",
                    "-fPIC", "-o", so, src], check=True, capture_output=True)
    lib = ctypes.CDLL(so)

    def call(f, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        assert lib.run(f, len(x), x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p)) == 0
        return y
    return call


def edges(lo, hi, n, rng):
    """Log-uniform magnitudes, and the mantissas where a seed changes binade."""
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    e = np.ldexp(1.0, rng.integers(-60, 60, 400))
    return np.concatenate([x, e, np.nextafter(e, 0), np.nextafter(e, np.inf), 3 * e, np.nextafter(2 * e, 0) * 0.5])


def worst(mp, got, x, exact):
    w = 0.0
    for g, v in zip(got, x):
        r = exact(mp.mpf(float(v)))
        w = max(w, float(abs(mp.mpf(float(g)) - r) / mp.mpf(float(np.spacing(abs(float(r)))))))
    return w


@pytest.mark.parametrize("f,bound", [(0, 0.51), (1, 1.0), (2, 0.51), (3, 1.1), (4, 1.1)],
                         ids=["rcp", "rsqrt", "sqrt", "exp", "half_erfc"])
def test_accuracy(run, f, bound):
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 50
    rng = np.random.default_rng(11 + f)
    if f <= 2:
        x = edges(1e-290, 1e290, 3000, rng)
        if f == 0:
            x = x * rng.choice([-1.0, 1.0], len(x))
        fn = [lambda v: 1 / v, lambda v: 1 / mp.sqrt(v), mp.sqrt][f]
    elif f == 3:
        x = np.concatenate([rng.uniform(-700, 700, 1500), rng.uniform(-3, 1, 1500), -np.exp(rng.uniform(-80, 0, 300)),
                            np.arange(-50, 50) * np.log(2) / 128, [0.0, -0.0]])
        fn = mp.exp
    else:
        k = np.arange(-143, 144) / 64.0
        x = np.concatenate([rng.uniform(-2.2499, 2.2499, 3000), k, np.nextafter(k, 9), np.exp(rng.uniform(-300, 0, 300)), [0.0]])
        fn = lambda v: mp.erfc(v) / 2
    assert worst(mp, run(f, x), x, fn) <= bound


def test_outside_the_fast_range(run):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, -1e-310, 1.7e308, -1.7e308, 2.3e-308])
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(run(0, x), 1.0 / x)
        np.testing.assert_allclose(run(1, x), 1.0 / np.sqrt(x), rtol=4e-16)
        np.testing.assert_array_equal(run(2, x), np.sqrt(x))
        e = np.array([-800.0, -745.0, -720.0, -701.0, 701.0, 709.0, 800.0, np.inf, -np.inf, np.nan])
        np.testing.assert_allclose(run(3, e), np.exp(e), rtol=1e-15, atol=5e-324)
        np.testing.assert_array_equal(run(5, x), (x > 0).astype(float))
        np.testing.assert_array_equal(run(6, x), np.fmin(x, 1.0))
