"""Reciprocal, reciprocal root and root of the FP64 collision (kernels.cuh)
against the exact values, and against CUDA's where they hand over to it."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1610_01388_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "kernels.cuh"
__global__ void k(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y[i] = blbm::moderate(x[i]) ? blbm::rcp(x[i]) : 0.0;
    y[n + i] = blbm::moderate(x[i]) ? blbm::rcp_root(x[i]) : 0.0;
    y[2 * n + i] = blbm::root(x[i]);
}
extern "C" int run(const double* x, double* y, int n) {
    double *dx = nullptr, *dy = nullptr;
    if (cudaMalloc(&dx, n * sizeof(double)) != cudaSuccess) return 1;
    if (cudaMalloc(&dy, 3 * n * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(dx, x, n * sizeof(double), cudaMemcpyHostToDevice);
    k<<<(n + 127) / 128, 128>>>(dx, dy, n);
    cudaMemcpy(y, dy, 3 * n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dy);
    return cudaGetLastError() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64")
    (d / "f.cu").write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-I", _build.CSRC, "-shared",
                    "-cudart", "static", str(d / "f.cu"), "-o", str(d / "f.so")], check=True)
    lib = ctypes.CDLL(str(d / "f.so"))

    def call(x):
        x = np.ascontiguousarray(x, np.float64)
        y = np.empty((3, x.size))
        p = ctypes.POINTER(ctypes.c_double)
        assert lib.run(x.ctypes.data_as(p), y.ctypes.data_as(p), ctypes.c_int(x.size)) == 0
        return y
    return call


def test_errors_in_ulps(functions):
    """Bounds from a start within 2^-18 (the hardware reads and gives 20 mantissa
    bits): 1 / x leaves e^3 <= 2^-54, half an ulp, and rounds once; 1 / sqrt(x)
    leaves 5/16 e^3 with e <= 2^-17, 1.25 ulp, half an ulp of the rounding in e
    and one rounding; the root adds a product."""
    r = np.random.default_rng(1)
    mantissa = np.concatenate([1.0 + r.random(3000), 2.0 - 2.0 ** -52 * np.arange(1, 9),
                               1.0 + 2.0 ** -52 * np.arange(9),
                               1.0 + 2.0 ** -20 * r.integers(0, 1 << 20, 500),
                               1.0 + 2.0 ** -20 * r.integers(1, 1 << 20, 500) - 2.0 ** -52])
    x = np.ldexp(mantissa, r.integers(-960, 960, mantissa.size))
    x = np.concatenate([x, [2.0 ** -960, np.nextafter(2.0 ** 960, 0.0)]])
    inverse, inverse_root, root = functions(x)
    worst = np.zeros(3)
    for i, a in enumerate(x):
        a = Fraction(float(a))
        for k, (v, bound) in enumerate(((inverse[i], 1.0), (inverse_root[i], 2.25), (root[i], 3.25))):
            got = Fraction(float(v))
            # relative error: of 1/x exactly, of the roots by halves of their squares'
            err = got * a - 1 if k == 0 else (got * got * a - 1) / 2 if k == 1 else (got * got / a - 1) / 2
            worst[k] = max(worst[k], abs(float(err * got / Fraction(float(np.spacing(v))))))
            assert worst[k] <= bound * (1 + 2.0 ** -10), (k, float(a))
    print("worst errors in ulps:", worst)


def test_root_outside_the_series(functions):
    x = np.array([0.0, 5e-324, 1e-310, 2.0 ** -1022, 1e-300, np.nextafter(2.0 ** -960, 0.0), 2.0 ** 960,
                  1e300, np.finfo(np.float64).max, np.inf])
    np.testing.assert_array_equal(functions(x)[2], np.sqrt(x))
    assert np.isnan(functions(np.array([np.nan]))[2][0])
