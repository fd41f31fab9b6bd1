"""DSum<float> (sums.cuh), the accumulator of the FP32 path's Lanczos sums: no less precise than an
FP64 sum of the same terms.

A kernel of one thread per row sums rows of floats; against the exact sum.  Tolerance: 2^-53 of
the sum (its conversion to double) and 2^-65 of the sum of the magnitudes (the third float's
roundings, at most 128 terms); a plain FP64 sum is allowed 2^-53 of the magnitudes per term."""
import ctypes
import math
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "sums.cuh"
__global__ void rows(const float* x, int n, double* out) {
  ll::DSum<float> s;
  for (int i = 0; i < n; ++i) s.add(x[blockIdx.x * n + i]);
  out[blockIdx.x] = s.value();
}
extern "C" int sums(const float* x, int nrow, int n, double* out) {
  float* dx; double* dout;
  if (cudaMalloc(&dx, sizeof(float) * nrow * n) != cudaSuccess || cudaMalloc(&dout, sizeof(double) * nrow) != cudaSuccess) return 1;
  cudaMemcpy(dx, x, sizeof(float) * nrow * n, cudaMemcpyHostToDevice);
  rows<<<nrow, 1>>>(dx, n, dout);
  cudaMemcpy(out, dout, sizeof(double) * nrow, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dout);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    from paper_2111_06623_gb300 import build
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.SRC,
                    "-o", str(d / "sums.so"), str(d / "sums.cu")], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "sums.so"))

    def run(x):
        out = np.zeros(len(x))
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert lib.sums(p(x), len(x), x.shape[1], p(out)) == 0
        return out
    return run


@pytest.mark.parametrize("n", [1, 2, 8, 32, 128])
@pytest.mark.parametrize("kind", ["positive", "signed", "cancelling", "decades"])
def test_no_less_precise_than_fp64(sums, n, kind):
    rng = np.random.default_rng(n)
    x = rng.normal(size=(200, n))
    if kind == "positive":
        x = abs(x)
    if kind == "decades":
        x *= 10.0 ** rng.uniform(-12, 0, x.shape)
    x = x.astype(np.float32)
    if kind == "cancelling" and n > 1:
        x[:, n // 2:] = -x[:, :n - n // 2] * (1 + np.float32(2.0 ** -22))
    got = sums(np.ascontiguousarray(x))
    for row, v in zip(x.astype(np.float64), got):
        exact, mag = math.fsum(row), math.fsum(abs(row))
        assert abs(v - exact) <= 2.0 ** -53 * abs(exact) + 2.0 ** -65 * mag


def test_not_finite(sums):
    x = np.ones((4, 3), np.float32)
    x[0, 1], x[1, 1], x[2, 1] = np.inf, -np.inf, np.nan
    got = sums(x)
    assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[2]) and got[3] == 3.0
