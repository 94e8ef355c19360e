"""The branch-free FP32 reciprocal, square root, quotient and inverse square root of the incident
field against IEEE arithmetic, over every mantissa, and the FP64 push's decisions by bits (zero, half,
one, floor of a move) against the comparisons they stand for: exact.

Tolerances.  One Newton step from an estimate of relative error e < 2^-22 leaves an error of at most
2^-44, so a result differs from the correctly rounded one only where the value lies within 2^-44 of
a rounding boundary, and then by one unit in the last place.  Boundaries are at most 2^-23 apart
(relative), so that happens for a fraction of 2 * 2^-44 / 2^-24 = 2^-19 of evenly spread arguments;
the bar is eight times that.  The inverse square root adds the rounding of its residual's product
(2^-24 e) and one final rounding: within one unit of the exact value."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_11393_gb300", "csrc")
SOURCE = r"""
#include "sff_common.cuh"
__global__ void k(int op, int n, const float* x, const float* y, float* r)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = op == 0 ? sff::m_inv(x[i]) : op == 1 ? sff::m_root(x[i]) : op == 2 ? sff::m_quot(y[i], x[i]) : sff::m_isqrt(x[i]);
}
__global__ void kb(int n, const double* x, int* r, double* f)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = sff::floor_unit(x[i], f[i]);
    r[i] = (k + 1) | (sff::nonzero(x[i]) << 4) | (sff::ge_half(x[i]) << 5) | (sff::ge_one(x[i]) << 6);
}
extern "C" int bits(int n, const double* x, int* r, double* f)
{
    char* d;
    if (cudaMalloc(&d, 20ll * n)) return 1;
    cudaMemcpy(d, x, 8ll * n, cudaMemcpyHostToDevice);
    kb<<<(n + 255) / 256, 256>>>(n, (const double*)d, (int*)(d + 16ll * n), (double*)(d + 8ll * n));
    cudaMemcpy(f, d + 8ll * n, 8ll * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(r, d + 16ll * n, 4ll * n, cudaMemcpyDeviceToHost);
    const int e = (int)cudaGetLastError();
    cudaFree(d);
    return e;
}
extern "C" int run(int op, int n, const float* x, const float* y, float* r)
{
    float* d;
    if (cudaMalloc(&d, 3ll * n * sizeof(float))) return 1;
    cudaMemcpy(d, x, 4ll * n, cudaMemcpyHostToDevice);
    cudaMemcpy(d + n, y, 4ll * n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(op, n, d, d + n, d + 2ll * n);
    cudaMemcpy(r, d + 2ll * n, 4ll * n, cudaMemcpyDeviceToHost);
    const int e = (int)cudaGetLastError();
    cudaFree(d);
    return e;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotients")
    (d / "q.cu").write_text(SOURCE)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC, "-shared",
                    "-Xcompiler", "-fPIC", "-o", str(d / "q.so"), str(d / "q.cu")], check=True, timeout=300)
    return ctypes.CDLL(str(d / "q.so"))


@pytest.mark.parametrize("exponent", [-20, -1, 0, 13])
@pytest.mark.parametrize("op", ["inv", "root", "quot", "isqrt"])
def test_every_mantissa(lib, op, exponent):
    n = 1 << 23
    x = ((np.uint32(127 + exponent) << np.uint32(23)) + np.arange(n, dtype=np.uint32)).view(np.float32)
    y = np.random.default_rng(5).uniform(2.0**-10, 2.0**10, n).astype(np.float32)
    r = np.empty_like(x)
    f = ctypes.POINTER(ctypes.c_float)
    k = ["inv", "root", "quot", "isqrt"].index(op)
    assert lib.run(k, n, x.ctypes.data_as(f), y.ctypes.data_as(f), r.ctypes.data_as(f)) == 0
    if op == "isqrt":
        exact = 1.0 / np.sqrt(x.astype(np.float64))
        assert (np.abs(r - exact) <= np.spacing(exact.astype(np.float32))).all()
        return
    want = np.float32(1) / x if op == "inv" else np.sqrt(x) if op == "root" else y / x
    off = np.abs(r.view(np.int32).astype(np.int64) - want.view(np.int32))
    assert off.max() <= 1
    assert np.count_nonzero(off) <= n * 2.0**-16


@pytest.mark.parametrize("op", ["inv", "root", "quot"])
def test_correctly_rounded(lib, op):
    """Not one unit off: every mantissa of an even and an odd exponent (the reciprocal and the root repeat
    beyond that), the quotient with a random numerator for each."""
    n = 1 << 24
    x = ((np.uint32(127) << np.uint32(23)) + np.arange(n, dtype=np.uint32)).view(np.float32)
    y = np.random.default_rng(7).uniform(1.0, 4.0, n).astype(np.float32)
    r = np.empty_like(x)
    f = ctypes.POINTER(ctypes.c_float)
    assert lib.run(["inv", "root", "quot"].index(op), n, x.ctypes.data_as(f), y.ctypes.data_as(f), r.ctypes.data_as(f)) == 0
    np.testing.assert_array_equal(r, np.float32(1) / x if op == "inv" else np.sqrt(x) if op == "root" else y / x)


def test_decisions_by_bits(lib):
    edges = np.array([-1.0, -0.5, 0.0, 0.5, 1.0, 2.0])
    x = np.concatenate([edges, np.nextafter(edges, 9), np.nextafter(edges, -9), [-0.0, 1e-310, -1e-310],
                        np.random.default_rng(6).uniform(-1, 2, 100001)])
    x = np.concatenate([x[(x >= -1) & (x < 2)], [np.nan, -np.nan]])
    r, fl = np.empty(len(x), np.int32), np.empty(len(x))
    p = ctypes.c_void_p
    assert lib.bits(len(x), x.ctypes.data_as(p), r.ctypes.data_as(p), fl.ctypes.data_as(p)) == 0
    k = np.nan_to_num(np.floor(x)).astype(int)
    np.testing.assert_array_equal((r & 15) - 1, k)
    np.testing.assert_array_equal(fl, k)
    np.testing.assert_array_equal((r >> 4) & 1, x != 0)
    np.testing.assert_array_equal((r >> 5) & 1, x >= 0.5)
    np.testing.assert_array_equal((r >> 6) & 1, x >= 1)
