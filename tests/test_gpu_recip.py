"""recip and recip_sqrt of the eigensolver and the Cholesky factor (csrc/recip.cuh, compiled here into a small program of its
own) against 1 / x and 1 / sqrt(x) in exact integer arithmetic: random mantissas over all exponents, powers of two and their
neighbours, and both sides of the exponents where they turn to the division.  Bound: the third-order step leaves about 2^-58
of the approximation's 2^-20, the residual and the final sum each round once: one unit in the last place, 2^-52 of the value."""
import ctypes
import os
import subprocess
from fractions import Fraction
from math import isqrt

import numpy as np
import pytest

from paper_1902_07455_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "recip.cuh"
__global__ void kernel(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = lrfg::recip(x[i]);
    s[i] = lrfg::recip_sqrt(fabs(x[i]));
  }
}
extern "C" int run(const double* x, double* r, double* s, int n) {
  double* d = nullptr;
  if (cudaMalloc(&d, 3 * sizeof(double) * n)) return 1;
  cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  kernel<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
  cudaMemcpy(r, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(s, d + 2 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("recip")
    (d / "recip.cu").write_text(SOURCE)
    out = str(d / "recip.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", build.CSRC, "-shared",
                    str(d / "recip.cu"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _inputs():
    rng = np.random.default_rng(7)
    e = np.concatenate([np.arange(1, 2047), np.repeat([1, 2, 22, 23, 24, 25, 1022, 1023, 2021, 2022, 2023, 2044, 2045], 200)])
    m = rng.integers(0, 1 << 52, e.size)
    m[:2046:5] = rng.choice([0, 1, (1 << 52) - 1], m[:2046:5].size)
    x = ((e.astype(np.uint64) << np.uint64(52)) | m.astype(np.uint64)).view(np.float64)
    x[::2] *= -1.0
    return x


def test_within_one_ulp(lib):
    x = np.ascontiguousarray(_inputs())
    r, s = np.empty_like(x), np.empty_like(x)
    p = [v.ctypes.data_as(ctypes.c_void_p) for v in (x, r, s)]
    assert lib.run(*p, x.size) == 0
    ulp = Fraction(1, 1 << 52)
    for xi, ri, si in zip(x, r, s):
        f = Fraction(float(xi))
        if abs(1.0 / xi) >= 2.0 ** -1022:
            assert abs(Fraction(float(ri)) * f - 1) <= ulp, xi
        # 1 / sqrt|x| to 2^-80 relative: floor(sqrt(2^(2 k) / |x|)) with a k that leaves some 90 bits
        k = 90 + int(np.frexp(xi)[1]) // 2
        q = (Fraction(4) ** k / abs(f))
        root = Fraction(isqrt(q.numerator // q.denominator)) / Fraction(2) ** k
        assert abs(Fraction(float(si)) / root - 1) <= ulp, xi
