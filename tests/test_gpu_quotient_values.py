"""The device functions behind the short quotients (common.cuh), called from a kernel
built here: against NumPy's division on ordinary values, at the ends of the range and
for infinities, NaN and zeros."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2001_11606_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
#include "common.cuh"
__global__ void run(int64_t n, const double *x, const double *d, double *q, double *b) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    q[i] = sphrt::quotient(x[i], d[i]);
    b[i] = sphrt::div_by(x[i], d[i], 1.0 / d[i]);
  }
}
extern "C" int quotients(int64_t n, const double *x, const double *d, double *q, double *b) {
  double *p = nullptr;
  const size_t nb = sizeof(double) * n;
  if (cudaMalloc(&p, 4 * nb) != cudaSuccess) return 1;
  cudaMemcpy(p, x, nb, cudaMemcpyHostToDevice);
  cudaMemcpy(p + n, d, nb, cudaMemcpyHostToDevice);
  run<<<256, 256>>>(n, p, p + n, p + 2 * n, p + 3 * n);
  cudaMemcpy(q, p + 2 * n, nb, cudaMemcpyDeviceToHost);
  cudaMemcpy(b, p + 3 * n, nb, cudaMemcpyDeviceToHost);
  const int rc = cudaGetLastError() != cudaSuccess;
  cudaFree(p);
  return rc;
}
"""


@pytest.fixture(scope="module")
def divide(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotients")
    src, lib = os.path.join(d, "q.cu"), os.path.join(d, "q.so")
    with open(src, "w") as fh:
        fh.write(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", "-o",
                    lib, src], check=True)
    L = C.CDLL(lib)

    def f(x, d):
        x, d = (np.ascontiguousarray(np.broadcast_to(a, np.broadcast(x, d).shape), dtype=np.float64)
                for a in (x, d))
        q, b = np.empty_like(x), np.empty_like(x)
        P = C.c_void_p
        assert L.quotients(C.c_int64(x.size), P(x.ctypes.data), P(d.ctypes.data),
                           P(q.ctypes.data), P(b.ctypes.data)) == 0
        return q, b, x, d
    return f


def _ulps(a, b):
    return np.abs(a - b) / np.spacing(np.minimum(np.abs(a), np.abs(b)))


def test_quotients_are_the_rounded_ones(divide):
    rng = np.random.default_rng(2)
    n = 1 << 20
    x = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-120, 121, n) * rng.choice([-1.0, 1.0], n)
    d = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(-120, 121, n) * rng.choice([-1.0, 1.0], n)
    q, b, x, d = divide(x, d)
    # the residual correction leaves ~2^-88 (2^-104 for div_by) before the final rounding:
    # about one value in 2^35 may round the other way, by one ulp
    for got in (q, b):
        off = _ulps(got, x / d)
        assert off.max() <= 1.0 and np.count_nonzero(off) <= 2


def test_ends_of_the_range(divide):
    tops = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e308, -1e308, 1.7e308, 1e-308, 5e-324, 1.0])
    bots = np.array([1.0, -3.0, 2.0 ** 99, 2.0 ** 100, 2.0 ** 101, 2.0 ** -99, 2.0 ** -100, 2.0 ** -101,
                     1e-300, 1e300])
    q, b, x, d = divide(tops[:, None], bots[None, :])
    with np.errstate(over="ignore"):
        want = x / d
    tiny = np.abs(want) < 2.0 ** -1000  # subnormal results: one unit of the smallest
    for got in (q, b):
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(np.isinf(got), np.isinf(want))
        fin = np.isfinite(want)
        assert np.array_equal(np.signbit(got[~fin & ~np.isnan(want)]),
                              np.signbit(want[~fin & ~np.isnan(want)]))
        tol = np.where(tiny, 5e-324, np.spacing(np.abs(np.where(fin, want, 1.0))))
        assert np.all(np.abs(got[fin] - want[fin]) <= tol[fin])


def test_division_by_zero_and_infinity(divide):
    x = np.array([1.0, -1.0, 0.0, np.inf, 1.0, -2.0, np.nan])
    d = np.array([0.0, 0.0, 0.0, 0.0, np.inf, -np.inf, 1.0])
    q = divide(x, d)[0]
    with np.errstate(divide="ignore", invalid="ignore"):
        assert np.array_equal(q, x / d, equal_nan=True)
