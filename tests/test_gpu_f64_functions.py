"""The FP64 building blocks by themselves, against CUDA's own functions and extended precision."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1801_03863_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "lbm_f64.cuh"
namespace {
template <int WHAT> __global__ void apply(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (WHAT == 0) y[i] = lbm::log1p_f64(x[i], 1.0 + x[i]);
    else if (WHAT == 1) y[i] = log1p(x[i]);
    else y[i] = lbm::rcp_f64(x[i]);
}
}
extern "C" int apply_f64(int what, const double* x, double* y, int n) {
    double* d = nullptr;
    if (cudaMalloc(&d, 2 * sizeof(double) * n)) return 1;
    cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    const int b = (n + 255) / 256;
    if (what == 0) apply<0><<<b, 256>>>(d, d + n, n);
    else if (what == 1) apply<1><<<b, 256>>>(d, d + n, n);
    else apply<2><<<b, 256>>>(d, d + n, n);
    const int e = (int)cudaMemcpy(y, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e;
}
"""
LOG, CUDA_LOG, RCP = 0, 1, 2


@pytest.fixture(scope="module")
def device_function(tmp_path_factory):
    folder = tmp_path_factory.mktemp("f64")
    (folder / "f.cu").write_text(SOURCE)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-I", _build.CSRC, "-shared",
                    "-o", str(folder / "f.so"), str(folder / "f.cu")], check=True)
    lib = ctypes.CDLL(str(folder / "f.so"))

    def call(what, x):
        y = np.empty_like(x)
        p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, y)]
        assert lib.apply_f64(what, *p, x.size) == 0
        return y
    return call


def _units(got, exact):
    """Relative errors in units of 2^-53."""
    return (np.abs((got - exact) / exact) * 2.0 ** 53).astype(np.float64)


@pytest.mark.parametrize("lo,hi", [(-0.75, 3.0), (-0.25, 0.25), (-0.0625, 0.0625)])
def test_logarithm_is_as_accurate_as_the_library(device_function, lo, hi):
    """Root mean square no more than 5 % above log1p's on the same values; at most one unit for the last
    rounding (a result just above a power of two), half a unit each for r and its polynomial next to y = 1,
    and an eighth for the table."""
    x = np.random.default_rng(1).uniform(lo, hi, 1 << 16)
    exact = np.log1p(x.astype(np.longdouble))
    table, library = (_units(device_function(w, x), exact) for w in (LOG, CUDA_LOG))
    assert table.max() <= 2.125
    assert np.sqrt((table ** 2).mean()) <= 1.05 * np.sqrt((library ** 2).mean())


def test_logarithm_outside_the_table(device_function):
    x = np.concatenate([np.array([-1.0, -2.0, 0.0, -0.0, np.inf, np.nan, 1e300, -1 + 2.0 ** -53, 3.0, 4.0]),
                        np.random.default_rng(2).uniform(3.0, 50.0, 1000),
                        np.random.default_rng(3).uniform(-1.0, -0.75, 1000)])
    a, b = device_function(LOG, x), device_function(CUDA_LOG, x)
    outside = (1.0 + x < 0.25) | (1.0 + x >= 4.0) | np.isnan(x)
    np.testing.assert_array_equal(a[outside], b[outside])
    assert (a[~outside] == b[~outside]).sum() >= 2  # the zeros


def test_reciprocal(device_function):
    """Error before the last rounding below 2^-65 of the result, so below half a unit in the last place
    and 2^-12 after it; outside FP32's range the IEEE quotient."""
    rng = np.random.default_rng(4)
    x = rng.uniform(1.0, 2.0, 1 << 18) * 2.0 ** rng.integers(-120, 120, 1 << 18) * rng.choice([-1.0, 1.0], 1 << 18)
    got = device_function(RCP, x)
    off = np.abs(got - 1 / x.astype(np.longdouble)) / np.abs(np.spacing(got))
    assert off.max() <= 0.5 + 2.0 ** -12
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, -1e-310, 1.7e308, -1.7e308, 1e300,
                     -1e-300, 2.0 ** 125, 2.0 ** -125, 2.0 ** 126, 2.0 ** -126, 2.0 ** 1022, 2.0 ** 1023])
    with np.errstate(divide="ignore", over="ignore"):
        np.testing.assert_array_equal(device_function(RCP, edge), 1.0 / edge)
