"""GPU: the double-float quotient, reciprocal, square root, inverse cube
root, exponential and logarithm as the device computes
them (the host tests compile the host branches, whose binary32 seeds are true
divisions and roots).  A small kernel over the library's header.

Bars, in units of u^2 = 2^-48, as the host tests': quotient 8, square root 4,
inverse cube root 6, e^x 4, ln 3 (of max(1, |ln x|)); the reciprocal as the
quotient."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U2 = 2.0 ** -48
SRC = r"""
#include "pointwise.cuh"
using namespace ofdft;
__global__ void k_ops(int op, int n, const double *x, const double *y, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const ff::f2 a = ff::from_double(x[i]), b = ff::from_double(y[i]);
    ff::f2 r(0.0f, 0.0f);
    switch (op) {
    case 0: r = ff::div(a, b); break;
    case 1: r = ff::recip(b); break;
    case 2: r = ff::sqrt(a); break;
    case 3: r = ff::rcbrt(a); break;
    case 4: r = ff::exp(a); break;
    case 5: r = ff::log(a); break;
    }
    out[i] = ff::to_double(r);
}
extern "C" int run(int op, int n, const double *x, const double *y, double *out)
{
    double *d = nullptr;
    if (cudaMalloc(&d, 3 * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(d, x, n * sizeof(double), cudaMemcpyHostToDevice);
    cudaMemcpy(d + n, y, n * sizeof(double), cudaMemcpyHostToDevice);
    k_ops<<<(n + 255) / 256, 256>>>(op, n, d, d + n, d + 2 * n);
    cudaMemcpy(out, d + 2 * n, n * sizeof(double), cudaMemcpyDeviceToHost);
    const int bad = cudaGetLastError() != cudaSuccess;
    cudaFree(d);
    return bad;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("ff")
    src, so = d / "ops.cu", d / "ops.so"
    src.write_text(SRC)
    csrc = os.path.join(ROOT, "paper_1406_0835_gb300", "csrc")
    subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                           "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I" + csrc, str(src), "-o", str(so),
                           "-lcudart"])
    lib = ctypes.CDLL(str(so))
    lib.run.argtypes = [ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 3

    def call(op, x, y):
        out = np.empty_like(x)
        assert lib.run(op, x.size, x.ctypes.data, y.ctypes.data, out.ctypes.data) == 0
        return out
    return call


def dd(x):
    """Nearest double-float of each binary64 (hi = float(x), lo = float(x - hi))."""
    hi = np.float32(x).astype(np.float64)
    return hi + np.float32(x - hi).astype(np.float64)


OPS = {   # reference in extended precision, operands' decades, bar
    "div": (0, lambda x, y: x / y, 12, 8.0),
    "recip": (1, lambda x, y: 1 / y, 12, 8.0),
    "sqrt": (2, lambda x, y: np.sqrt(x), 18, 4.0),
    "rcbrt": (3, lambda x, y: 1 / np.cbrt(x), 18, 6.0),
    "exp": (4, lambda x, y: np.exp(x), None, 4.0),
    "log": (5, lambda x, y: np.log(x), 25, 3.0),
}


@pytest.mark.parametrize("op", OPS)
def test_device_operations(run, op):
    code, ref, decades, bar = OPS[op]
    rng = np.random.default_rng(code)
    n = 200000
    if decades is None:
        x = dd(rng.uniform(-60.0, 60.0, n))
    else:
        x = dd(10.0 ** rng.uniform(-decades, decades, n))
    y = dd(rng.uniform(0.5, 1.0, n) * 10.0 ** rng.uniform(-12, 12, n))
    if code < 2:
        x *= np.where(rng.random(n) < 0.5, -1.0, 1.0)
        y *= np.where(rng.random(n) < 0.5, -1.0, 1.0)
    want = ref(np.longdouble(x), np.longdouble(y))
    got = run(code, x, y)
    scale = np.maximum(1, np.abs(want)) if op == "log" else np.abs(want)
    err = np.abs(np.longdouble(got) - want) / scale / U2
    print(op, "rms %.3f max %.2f" % (float(np.sqrt(np.mean(err ** 2))), float(err.max())))
    assert err.max() < bar
