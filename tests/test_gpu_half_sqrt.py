"""The square root of the FP64 face flux (half_sqrt in csrc/arith.cuh), compiled into a kernel of
its own: rounded like the IEEE square root over the whole range of FP64, with its special values.

Tolerance: half a unit in the last place for the rounding, and 2^-10 of a unit for what the
reference (extended precision) and the last correction leave (2^-11 and 2^-33).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

SOURCE = """
#include "arith.cuh"
__global__ void roots(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = adg::half_sqrt(x[i]);
}
extern "C" int run(const double* x, double* y, int n) {
  double *dx, *dy;
  const size_t b = sizeof(double) * n;
  if (cudaMalloc(&dx, b) || cudaMalloc(&dy, b)) return 1;
  cudaMemcpy(dx, x, b, cudaMemcpyHostToDevice);
  roots<<<(n + 255) / 256, 256>>>(dx, dy, n);
  const cudaError_t e = cudaMemcpy(y, dy, b, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2603_28710_gb300 import build as b
    d = tmp_path_factory.mktemp("sqrt")
    src, lib = str(d / "roots.cu"), str(d / "roots.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-shared", "-o", lib, src], check=True, cwd=ROOT)
    fn = ctypes.CDLL(lib).run

    def call(x):
        x = np.ascontiguousarray(x, np.float64)
        y = np.empty_like(x)
        assert fn(x.ctypes.data_as(ctypes.c_void_p), y.ctypes.data_as(ctypes.c_void_p), x.size) == 0
        return y
    return call


@pytest.mark.parametrize("lo,hi", [(0, 2), (-2, 0), (-1021, 1023)])
def test_rounding(roots, lo, hi):
    rng = np.random.default_rng((lo + 7) % 2 ** 32)
    x = np.ldexp(rng.uniform(0.5, 1.0, 1 << 20), rng.integers(lo + 1, hi + 1, 1 << 20))
    x = np.concatenate([x, np.nextafter(2.0 ** np.arange(lo + 1, hi), 0.0), 2.0 ** np.arange(lo, hi)])
    ref = np.sqrt(x.astype(np.longdouble)) / 2
    y = roots(x)
    ulp = np.spacing(np.asarray(ref, np.float64))
    err = np.abs(y - ref) / ulp
    assert err.max() <= 0.5 + 2.0 ** -10, float(err.max())


def test_special_values(roots):
    tiny = 2.0 ** -1074
    x = np.array([0.0, -0.0, tiny, 3 * tiny, 2.0 ** -1022, np.inf, -np.inf, -1.0, np.nan,
                  np.finfo(np.float64).max])
    with np.errstate(invalid="ignore"):
        assert np.array_equal(roots(x), 0.5 * np.sqrt(x), equal_nan=True)
