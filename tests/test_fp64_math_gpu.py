"""The short FP64 functions of csrc/fp64_math.cuh against long double on the host.

Bounds from the series and seeds: the Householder steps leave (2^-20)^3 relative, the logarithm's series r^9/9 at
|r| <= 2^-7, the arctangent's z^9/9 at |z| <= 2^-7, Taylor remainders (pi/4)^17/17!; with one rounding per
operation on results of order one each stays within 4 units of 2^-53 of max(1, |value|) -- relative for the reciprocal
forms and for the logarithm near 1, absolute 2^-51 for sine and cosine.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "%s/paper_2111_11058_gb300/csrc/fp64_math.cuh"
using namespace cbfm::f64;
__global__ void k(int n, const double *x, const double *y, double *o) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    o[i] = rcp64(x[i]);
    o[n + i] = rsqrt64(x[i]);
    o[2 * n + i] = log64(x[i]);
    o[3 * n + i] = atan2_pos(x[i], y[i]);
    sincos64(y[i], &o[4 * n + i], &o[5 * n + i]);
}
extern "C" int run(int n, const double *x, const double *y, double *o) {
    double *dx, *dy, *d;
    cudaMalloc(&dx, 8 * n); cudaMalloc(&dy, 8 * n); cudaMalloc(&d, 48 * n);
    cudaMemcpy(dx, x, 8 * n, cudaMemcpyHostToDevice); cudaMemcpy(dy, y, 8 * n, cudaMemcpyHostToDevice);
    k<<<(n + 127) / 128, 128>>>(n, dx, dy, d);
    const int e = cudaMemcpy(o, d, 48 * n, cudaMemcpyDeviceToHost);
    cudaFree(dx); cudaFree(dy); cudaFree(d);
    return e;
}
"""


def test_against_long_double(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_11058_gb300 import build as B
    cu, so = str(tmp_path / "f.cu"), str(tmp_path / "f.so")
    with open(cu, "w") as f:
        f.write(SRC % ROOT)
    subprocess.run([B.nvcc(), "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", *B.ARCH, cu, "-o", so], check=True)
    rng = np.random.default_rng(3)
    edge = np.concatenate([[1.0, 0.75, 1.5, 2.0, 0.5, 1e-30, 1e30, 3.0], 1.0 + 2.0 ** -np.arange(1, 53.0),
                           1.0 - 2.0 ** -np.arange(2, 53.0), 0.75 + np.arange(64) / 256.0, 1.0 + np.arange(64) / 128.0])
    x = np.concatenate([edge, np.exp(rng.uniform(-40, 40, 200000)), rng.uniform(0.5, 2.0, 100000)])
    y = np.concatenate([np.tile([0.0, 1.0, -1.0, np.pi / 4, -np.pi / 2, 1e4, 2e5, -99999.0], len(edge))[:len(edge)],
                        np.exp(rng.uniform(-40, 11, 200000)) * rng.choice([-1, 1], 200000), rng.uniform(-2, 2, 100000)])
    n = len(x)
    o = np.zeros((6, n))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    assert ctypes.CDLL(so).run(n, p(x), p(y), p(o)) == 0
    X, Y = x.astype(np.longdouble), y.astype(np.longdouble)
    u = 2.0 ** -53
    rel = lambda a, r: float(np.max(np.abs(a - r) / np.abs(r)))  # noqa: E731
    assert rel(o[0], 1 / X) <= 4 * u
    assert rel(o[1], 1 / np.sqrt(X)) <= 4 * u
    r = np.log(X)
    near = np.abs(x - 1) < 2.0 ** -8
    assert np.max(np.abs(o[2] - r) / np.maximum(1, np.abs(r))) <= 4 * u
    assert (np.abs(o[2] - r)[near] <= 4 * u * np.abs(r)[near]).all()
    assert np.max(np.abs(o[3] - np.arctan2(X, Y))) <= 8 * u
    small = X < np.abs(Y) / 128
    small &= y > 0
    assert (np.abs(o[3] - np.arctan2(X, Y))[small] <= 8 * u * np.arctan2(X, Y)[small]).all()
    assert np.max(np.abs(o[4] - np.sin(Y))) <= 4 * u and np.max(np.abs(o[5] - np.cos(Y))) <= 4 * u
