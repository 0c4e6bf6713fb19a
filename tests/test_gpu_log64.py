"""The binary64 logarithm and reciprocal of the kernels (lbm_core.cuh) against extended
precision, beside CUDA's log and division on the same arguments.

Bounds.  log64: the last addition rounds once (half an ulp of the result); before it,
|r^5 - 0.87 2^-22 r^3| / 5 <= 0.13 2^-55 / 5 of the polynomial, r^6 / 6 <= 2^-68, one
rounding of a sum below 2^-11 (2^-65) and the low words of the tables (2^-67 each):
8e-19 together.  rcp64: the seed is good to 2^-20, so the series cut after the square
leaves 2^-60 before the last operation, which rounds once: half an ulp and 2^-6 of one.
"""
from __future__ import annotations

import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "lbm_core.cuh"
using namespace lbmfug;
__global__ void k(const double *x, int n, const Log64 *t, double *l, double *lc, double *r, double *rc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    l[i] = log64(x[i], t);
    lc[i] = log(x[i]);
    r[i] = rcp64(x[i]);
    rc[i] = 1.0 / x[i];
}
extern "C" int run(const double *x, int n, double *out)
{
    double *d = nullptr;
    Log64 *t = nullptr;
    if (cudaMalloc(&d, 5 * sizeof(double) * n) != cudaSuccess || cudaMalloc(&t, sizeof(Log64)) != cudaSuccess) return 1;
    int e = cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    if (!e) e = cudaMemcpy(t, &log64_host(), sizeof(Log64), cudaMemcpyHostToDevice);
    if (!e) {
        k<<<(n + 255) / 256, 256>>>(d, n, t, d + n, d + 2 * n, d + 3 * n, d + 4 * n);
        e = cudaMemcpy(out, d + n, 4 * sizeof(double) * n, cudaMemcpyDeviceToHost);
    }
    cudaFree(d);
    cudaFree(t);
    return e;
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    from paper_2306_10652_gb300 import build as b
    d = tmp_path_factory.mktemp("log64")
    (d / "k.cu").write_text(SRC)
    so = d / "k.so"
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-shared", str(d / "k.cu"), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))

    def f(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        out = np.empty((4, x.size))
        p = ctypes.POINTER(ctypes.c_double)
        assert lib.run(x.ctypes.data_as(p), x.size, out.ctypes.data_as(p)) == 0
        return out

    return f


RANGES = [(1e-300, 1e-290), (1e-8, 1e-4), (1e-4, 0.01), (0.01, 0.5), (0.5, 0.9), (0.9, 1.0), (1.0 - 2.0**-11, 1.0),
          (1.0, 1.1), (1.0, 20.0), (1e290, 1e300)]


@pytest.mark.parametrize("lo,hi", RANGES, ids=lambda v: f"{v:.3g}")
def test_log64_is_as_accurate_as_the_library(evaluate, lo, hi):
    x = np.random.default_rng(7).uniform(lo, hi, 200000)
    got, lib = evaluate(x)[:2]
    ref = np.log(x.astype(np.longdouble))
    e = np.abs(got - ref).astype(np.float64)
    assert (e <= 0.5 * np.spacing(np.abs(ref).astype(np.float64)) + 8e-19).all(), e.max()
    el = np.abs(lib - ref).astype(np.float64)
    assert np.sqrt((e**2).mean()) <= 1.02 * np.sqrt((el**2).mean()) + 8e-19


@pytest.mark.parametrize("lo,hi", RANGES, ids=lambda v: f"{v:.3g}")
def test_rcp64_rounds_once(evaluate, lo, hi):
    x = np.random.default_rng(8).uniform(lo, hi, 200000)
    got = evaluate(np.concatenate([x, -x]))[2]
    ref = np.longdouble(1) / np.concatenate([x, -x]).astype(np.longdouble)
    e = np.abs(got - ref).astype(np.float64)
    assert (e <= (0.5 + 2.0**-6) * np.spacing(np.abs(got))).all()


def test_special_arguments(evaluate):
    tiny, big = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    # zeros, infinities, NaN and exact reciprocals as the division gives them
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.0, -1.0, 0.5, -2.0, tiny, -tiny, 2.0**1021, 2.0**1022])
    _, _, r, rc = evaluate(x)
    assert np.array_equal(r, rc, equal_nan=True) and np.array_equal(np.signbit(r), np.signbit(rc))
    # subnormal arguments count as zeros, subnormal results may be
    assert np.array_equal(evaluate([5e-324, tiny / 3, -tiny / 3])[2], [np.inf, np.inf, -np.inf])
    assert (np.abs(evaluate([big, -big, 2.0**1023])[2]) < tiny).all()
    # log64: the library's log where the table does not reach, and ln 1 to the part before the
    # last addition
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, 5e-324, tiny / 3])
    l, lc, _, _ = evaluate(x)
    assert np.array_equal(l, lc, equal_nan=True)
    l, lc, _, _ = evaluate([1.0, 0.5, 2.0, 1024.0])
    assert abs(l[0]) <= 8e-19 and np.array_equal(l[1:], lc[1:])
