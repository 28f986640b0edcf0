"""rcp_h3 and rsqrt_h3 (fix.cuh) against their stated 2 ulp, over random mantissas and the exponents whose
results are normal, both signs for the reciprocal (pivots are often negative); 0, denormals and infinities
give no finite number, and NaN gives NaN."""
import ctypes

import numpy as np
import pytest

from tests.cuda_helper import compile_cuda

pytestmark = pytest.mark.gpu

SOURCE = r'''
#include "fix.cuh"
__global__ void k(int n, const double* x, double* r, double* q) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = emg::rcp_h3(x[i]), q[i] = emg::rsqrt_h3(x[i]);
}
extern "C" int unit(int n, const double* x, double* r, double* q) {
    double* d = nullptr;
    if (cudaMalloc(&d, (size_t)3 * n * 8) != cudaSuccess) return 1;
    cudaMemcpy(d, x, (size_t)n * 8, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(n, d, d + n, d + 2 * n);
    cudaMemcpy(r, d + n, (size_t)n * 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(q, d + 2 * n, (size_t)n * 8, cudaMemcpyDeviceToHost);
    const int e = (int)cudaGetLastError();
    cudaFree(d);
    return e;
}
'''


@pytest.fixture(scope="module")
def unit(tmp_path_factory):
    lib = compile_cuda(SOURCE, str(tmp_path_factory.mktemp("reciprocals")))

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        r, q = np.empty_like(x), np.empty_like(x)
        p = [ctypes.c_void_p(a.ctypes.data) for a in (x, r, q)]
        assert lib.unit(ctypes.c_int(x.size), *p) == 0
        return r, q
    return call


def ulps(a, b):
    """|a - b| in units of the last place of b (b given with more bits)."""
    return np.abs((a.astype(np.longdouble) - b) / np.spacing(np.abs(b.astype(np.float64)))).astype(float)


@pytest.mark.parametrize("lo,hi", [(-3, 3), (-300, 300), (-1020, 1020)])
def test_within_two_ulp(unit, lo, hi):
    rng = np.random.default_rng(hi)
    x = np.ldexp(rng.uniform(1.0, 2.0, 1 << 20), rng.integers(lo, hi, 1 << 20))
    x[:4096] = np.ldexp(np.nextafter(np.repeat([1.0, 2.0], 2048), 0.0), rng.integers(lo, hi, 4096))
    exact = x.astype(np.longdouble)
    r, q = unit(x)
    assert ulps(r, 1 / exact).max() <= 2
    assert ulps(q, 1 / np.sqrt(exact)).max() <= 2
    np.testing.assert_array_equal(unit(-x)[0], -r)


def test_no_number_from_none(unit):
    r, q = unit(np.array([0.0, -0.0, 5e-324, 1e-310, np.inf, -np.inf, np.nan]))
    assert not np.isfinite(r).any() and not np.isfinite(q).any()
    assert np.isnan(unit(np.array([-1.0, -1e-300, -np.inf]))[1]).all()
