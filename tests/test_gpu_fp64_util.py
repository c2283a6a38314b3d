"""rcp64 and rsqrt64 (csrc/fp64_util.h) over the whole exponent range, compiled into
a small kernel of their own: against exact rational arithmetic within 0.6 and 1.1
ulp (the roundings of their last operations), and where the FP32 range does not
hold the exponent, and at zero, infinity and NaN, the same bits as CUDA's."""
import ctypes as C
import math
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import gpu_lib

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fp64_util.h"
__global__ void k(const double* x, int n, double* r, double* s, double* cr, double* cs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = ofm::rcp64(x[i]);
  s[i] = ofm::rsqrt64(x[i]);
  cr[i] = 1.0 / x[i];
  cs[i] = rsqrt(x[i]);
}
extern "C" int run(const double* x, int n, double* out) {
  double* d = nullptr;
  const size_t b = sizeof(double) * n;
  if (cudaMalloc(&d, 5 * b) != cudaSuccess) return 1;
  cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, n, d + n, d + 2 * n, d + 3 * n, d + 4 * n);
  const cudaError_t e = cudaMemcpy(out, d + n, 4 * b, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def util(tmp_path_factory):
    gpu_lib()
    from paper_1011_4764_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    (d / "k.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", *build.ARCH,
                    "-I", build.CSRC, str(d / "k.cu"), "-o", str(d / "k.so")], check=True)
    lib = C.CDLL(str(d / "k.so"))

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        out = np.empty((4, x.size))
        p = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
        assert lib.run(p(x), x.size, p(out)) == 0
        return out
    return run


def _arguments():
    rng = np.random.default_rng(3)
    m = np.concatenate([1.0 + rng.random(3), [1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0)]])
    return np.concatenate([np.ldexp(m, e) for e in range(-1021, 1021, 7)] + [np.ldexp(m, e) for e in (-101, -100, -99, -98, 98, 99, 100, 101)])


def test_rounding_over_the_range(util):
    x = _arguments()
    r, s, _, _ = util(x)
    for v, a, b in zip(x, r, s):
        q = 1 / Fraction(v)
        assert abs(Fraction(float(a)) - q) <= Fraction(6, 10) * Fraction(math.ulp(float(a))), v
        # |b - x^-1/2| <= t: (b - t)^2 x <= 1 <= (b + t)^2 x
        t = Fraction(11, 10) * Fraction(math.ulp(float(b)))
        lo, hi = Fraction(float(b)) - t, Fraction(float(b)) + t
        assert lo * lo * Fraction(v) <= 1 <= hi * hi * Fraction(v), v


def test_outside_the_range_as_cuda(util):
    tiny = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, -1e-310, 2.0 ** -1022, 1.7e308, -1.7e308,
                     2.0 ** -120, 2.0 ** 120, -(2.0 ** 300)])
    r, s, cr, cs = util(tiny)
    for a, b in ((r, cr), (s, cs)):
        assert np.array_equal(np.isnan(a), np.isnan(b))
        keep = ~np.isnan(a)
        assert np.array_equal(a[keep].view(np.int64), b[keep].view(np.int64))


def test_negative_arguments(util):
    x = -_arguments()
    r, s, _, _ = util(x)
    assert np.array_equal(r, -util(-x)[0]) and np.all(np.isnan(s))
