"""FP64 reciprocal and square root of the step (csrc/lbm_internal.cuh), from the
hardware seeds (relative error about 2^-20) and two terms of the series, against
1/x and sqrt(x) in extended precision.  What the series leaves out is of order
2^-60, 0.01 ulp.  The reciprocal adds the rounding of its last operation: 0.51
ulp.  The square root adds half of the rounding of x y, which its correction
takes for a part of the seed's error: 0.76 ulp."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "lbm_internal.cuh"
__global__ void k_eval(const double* x, double* r, double* s, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = lbm::f_rcp(x[i]);
    s[i] = lbm::f_sqrt(x[i]);
}
extern "C" int eval(const double* x, double* r, double* s, long long n) {
    double* d = nullptr;
    const size_t b = (size_t)n * sizeof(double);
    if (cudaMalloc(&d, 3 * b) != cudaSuccess) return 1;
    cudaError_t e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_eval<<<(unsigned)((n + 255) / 256), 256>>>(d, d + n, d + 2 * n, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(r, d + n, b, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(s, d + 2 * n, b, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    from paper_2205_00686_gb300 import _build as B
    d = tmp_path_factory.mktemp("math")
    src, so = str(d / "eval.cu"), str(d / "eval.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I" + B.CSRC, "-shared", src, "-o", so], check=True)
    L = ctypes.CDLL(so)

    def run(x):
        x = np.ascontiguousarray(x, np.float64)
        r, s = np.empty_like(x), np.empty_like(x)
        p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, r, s)]
        assert L.eval(*p, ctypes.c_longlong(x.size)) == 0
        return r, s
    return run


def ulps(got, exact):
    """Distance in units of the last place of the double nearest to `exact`."""
    return float((np.abs(got.astype(np.longdouble) - exact) / np.spacing(exact.astype(np.float64))).max())


def test_within_the_derived_bounds(evaluate):
    rng = np.random.default_rng(1)
    # what the step feeds them (densities, 1 - b rho, T / T_c, psi^2), every
    # mantissa of one binade coarsely, and numbers next to powers of two
    x = np.concatenate([np.exp(rng.uniform(np.log(1e-6), np.log(1e3), 400000)),
                        1.0 + np.arange(200000) / 200000.0, 2.0 + np.arange(200000) / 100000.0,
                        np.nextafter(2.0 ** np.arange(-30, 31), 0.0), 2.0 ** np.arange(-30, 31),
                        np.nextafter(2.0 ** np.arange(-30, 31), np.inf)])
    r, s = evaluate(x)
    xl = x.astype(np.longdouble)
    assert ulps(r, np.longdouble(1) / xl) <= 0.51
    assert ulps(s, np.sqrt(xl)) <= 0.76


def test_square_root_over_the_whole_range(evaluate):
    rng = np.random.default_rng(2)
    # both ends of the fast range, 2^-1000 and 2^1000, from either side
    ends = [np.nextafter(e, t) for e in (2.0 ** -1000, 2.0 ** 1000) for t in (0.0, e, np.inf)]
    x = np.concatenate([2.0 ** rng.uniform(-1074, 1023.9, 200000), ends,
                        [5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0.0), np.finfo(float).max]])
    assert ulps(evaluate(x)[1], np.sqrt(x.astype(np.longdouble))) <= 0.76
    s = evaluate(np.array([0.0, -0.0, np.inf, -1.0, -5e-324, -np.inf, np.nan]))[1]
    assert s[0] == 0.0 and s[1] == 0.0 and s[2] == np.inf and np.isnan(s[3:]).all()


def test_reciprocal_of_unusable_operands_is_not_finite(evaluate):
    r = evaluate(np.array([0.0, -0.0, np.inf, -np.inf, np.nan]))[0]
    assert not np.isfinite(r).any()
