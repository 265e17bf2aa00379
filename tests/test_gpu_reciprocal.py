"""The reciprocal of the density that every update, capture, rebuild and
restriction divides by (vrcp of csrc/lattice.cuh), compiled as it stands there:
correctly rounded, so equal bit for bit to the binary32 division of the host
-- every density of two binades around one and of other binades, and the ends
of the range (zero, infinity, NaN, subnormal numbers) -- one value at a time and
in the two lanes of the packed arithmetic."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lattice.cuh"
using namespace mlbm;
__global__ void k_one(const float* x, float* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = vrcp(x[i]);
}
__global__ void k_two(const float2* x, float2* r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = vrcp(F2{x[i]}).v;
}
extern "C" int reciprocal(const float* x, float* one, float* two, int n) {  // n even
  float *dx = nullptr, *dr = nullptr;
  const size_t bytes = sizeof(float) * (size_t)n;
  cudaError_t e = cudaMalloc(&dx, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&dr, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(dx, x, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_one<<<(n + 127) / 128, 128>>>(dx, dr, n);
    e = cudaMemcpy(one, dr, bytes, cudaMemcpyDeviceToHost);
  }
  if (e == cudaSuccess) {
    k_two<<<(n / 2 + 127) / 128, 128>>>((const float2*)dx, (float2*)dr, n / 2);
    e = cudaMemcpy(two, dr, bytes, cudaMemcpyDeviceToHost);
  }
  cudaFree(dx);
  cudaFree(dr);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def reciprocal(tmp_path_factory):
    from paper_2004_11863_gb300 import build

    d = tmp_path_factory.mktemp("reciprocal")
    src, lib = d / "reciprocal.cu", d / "libreciprocal.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, f"-I{build.CSRC}", "-shared",
                    "-o", str(lib), str(src), "-lcudart"], check=True)
    f = ctypes.CDLL(str(lib)).reciprocal

    def call(x):
        one, two = np.empty_like(x), np.empty_like(x)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert f(p(x), p(one), p(two), x.size) == 0
        return one, two

    return call


def check(reciprocal, x):
    with np.errstate(divide="ignore", over="ignore", invalid="ignore"):
        want = np.float32(1.0) / x
    for got in reciprocal(x):
        nan = np.isnan(want)
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got[~nan].view(np.uint32), want[~nan].view(np.uint32))


@pytest.mark.parametrize("exponent", [-126, -125, -40, -1, 0, 40, 125, 126, 127])
def test_correctly_rounded(reciprocal, exponent):
    x = np.arange((exponent + 127) << 23, (exponent + 128) << 23, dtype=np.uint32)
    check(reciprocal, x.view(np.float32))


def test_ends_of_the_range(reciprocal):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-45, -1e-45, 1e-39, 2.0 ** -128, 2.0 ** -129,
                  -1.0, 3.4e38], dtype=np.float32)
    check(reciprocal, x)
