"""The gate functions of the sequential loop's rolled phase A (sigmoid_nb, tanh_nb) are as accurate as the
library's 1 / (1 + expf(-x)) and tanhf: over every fp32 argument of a run of intervals, the largest error
against fp64, in units of the last place, is no larger than the library's on the same interval and
within a bound of its own.  The kernel under test is a loop over the functions, compiled here from the
header that the loop's kernels include.

The bounds.  sigmoid: expf within 2 units (its documented bound: 2.4e-7 relative), the sum and the
refined reciprocal half a unit each (6e-8): 3.6e-7 of the value, at most 6 units of its last place.
tanh from 1 on: 1 - 2 / (1 + e^2x), where the subtracted term is at most 0.24, so its 3.6e-7 come to
8.6e-8 = 1.5 units, and the rounding of the result adds half a one: 2.  Below 1, x + x s t(s): the
correction is at most 0.31 of the value, its rounding errors (s, x s, t: 1.5 units each of 6e-8) and
the truncation of t (0.2) come to 0.31 * 4.7 = 1.5 units, and half a one again: 2.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2605_29707_gb300 import build as _build

pytestmark = pytest.mark.gpu

# (0.5, 0.51) and (1, 1.01): just past where the two forms of tanh have met
EDGES = np.array([2.0**-20, 2.0**-6, 0.25, 0.49, 0.5, 0.51, 0.625, 0.75, 0.875, 0.99, 1.0, 1.01, 1.125, 1.25, 1.5, 2.0,
                  4.0, 9.0, 20.0, 40.0, 80.0], np.float32)

SOURCE = r"""
#include "rollout_kernels.cuh"
template <int F> __device__ float value(float x) {
  if (F == 0) return dm::tanh_nb(x);
  if (F == 1) return tanhf(x);
  if (F == 2) return dm::sigmoid_nb(x);
  return 1.f / (1.f + expf(-x));
}
// *err = 1024 x the largest error of F over the floats lo <= |x| < hi (bit patterns), in units of the last place
template <int F> __global__ void scan(uint32_t lo, uint32_t hi, uint32_t sign, unsigned long long* err) {
  unsigned long long worst = 0;
  for (unsigned long long u = lo + blockIdx.x * 256ull + threadIdx.x; u < hi; u += gridDim.x * 256ull) {
    const float x = __uint_as_float(static_cast<uint32_t>(u) | sign);
    const double xd = x, ref = F < 2 ? tanh(xd) : 1.0 / (1.0 + exp(-xd));
    int e;
    frexp(ref, &e);
    const double d = fabs(static_cast<double>(value<F>(x)) - ref) * ldexp(1.0, 24 - e);
    const unsigned long long w = d < 1e9 ? static_cast<unsigned long long>(d * 1024.0) : 1ull << 40;
    worst = w > worst ? w : worst;
  }
  atomicMax(err, worst);
}
template <int F> __global__ void at(const float* x, float* y, int n) {
  if (static_cast<int>(threadIdx.x) < n) y[threadIdx.x] = value<F>(x[threadIdx.x]);
}
template <int F> static int run(uint32_t lo, uint32_t hi, uint32_t sign, double* out) {
  unsigned long long* d = nullptr;
  unsigned long long h = 0;
  if (cudaMalloc(&d, 8) != cudaSuccess) return 1;
  cudaMemset(d, 0, 8);
  scan<F><<<608, 256>>>(lo, hi, sign, d);
  const cudaError_t e = cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
  cudaFree(d);
  *out = static_cast<double>(h) / 1024.0;
  return e != cudaSuccess;
}
extern "C" __attribute__((visibility("default"))) int gates_worst(int f, uint32_t lo, uint32_t hi, uint32_t sign, double* out) {
  if (f == 0) return run<0>(lo, hi, sign, out);
  if (f == 1) return run<1>(lo, hi, sign, out);
  if (f == 2) return run<2>(lo, hi, sign, out);
  return run<3>(lo, hi, sign, out);
}
extern "C" __attribute__((visibility("default"))) int gates_at(int f, const float* x, float* y, int n) {  // n <= 256, host memory
  float *dx = nullptr, *dy = nullptr;
  if (n > 256 || cudaMalloc(&dx, 1024) != cudaSuccess || cudaMalloc(&dy, 1024) != cudaSuccess) return 1;
  cudaMemcpy(dx, x, n * 4, cudaMemcpyHostToDevice);
  if (f == 0) at<0><<<1, 256>>>(dx, dy, n);
  else at<2><<<1, 256>>>(dx, dy, n);
  const cudaError_t e = cudaMemcpy(y, dy, n * 4, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  return e != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("gates")
    src, so = str(d / "gates.cu"), str(d / "gates.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    cmd = [_build.nvcc()] + _build._flags() + ["-shared", "-cudart", "static", "-o", so, src]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert os.path.exists(so)
    return ctypes.CDLL(so)


def _worst(lib, f, lo, hi, negative):
    bits = np.array([lo, hi], np.float32).view(np.uint32)
    out = ctypes.c_double()
    assert lib.gates_worst(f, ctypes.c_uint32(int(bits[0])), ctypes.c_uint32(int(bits[1])),
                           ctypes.c_uint32(0x80000000 if negative else 0), ctypes.byref(out)) == 0
    return out.value


@pytest.mark.parametrize("negative", [False, True], ids=["positive", "negative"])
@pytest.mark.parametrize("fast,library,bound", [(0, 1, 2.0), (2, 3, 6.0)], ids=["tanh", "sigmoid"])
def test_gate_functions_are_as_accurate_as_the_library(lib, fast, library, bound, negative):
    for lo, hi in zip(EDGES[:-1], EDGES[1:]):
        a, b = _worst(lib, fast, lo, hi, negative), _worst(lib, library, lo, hi, negative)
        assert a <= b and a <= bound, (float(lo), float(hi), a, b)


def test_gate_functions_at_the_ends(lib):
    inf = np.float32(np.inf)
    x = np.array([0.0, -0.0, 1e-40, 40.0, -40.0, 100.0, -100.0, 3e38, -3e38, inf, -inf, np.nan], np.float32)
    y = np.empty_like(x)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    assert lib.gates_at(0, ptr(x), ptr(y), len(x)) == 0
    np.testing.assert_array_equal(y, np.tanh(x.astype(np.float64)).astype(np.float32))
    assert lib.gates_at(2, ptr(x), ptr(y), len(x)) == 0
    with np.errstate(over="ignore"):
        ref = 1.0 / (1.0 + np.exp(-x.astype(np.float64)))
    # far below zero the smallest value is e^-87, past which the difference is under 2e-38
    np.testing.assert_allclose(y, ref, rtol=3.6e-7, atol=2e-38)
