"""GPU: one transform of k_tline by itself, against the matrix product in
extended precision.

Bar: the root mean square of (error / one standard deviation) stays below 2.
One deviation of an output, in units of its line's largest value times the
largest matrix entry: the dropped products of digits, six for each of the n
terms, each 74^2 rms (digits of radix 256) of weight 2^40 against at least 2^52
and 2^53, so sqrt(6 n) 2^-52.6; the rounding of line and matrix, sqrt(n)
2^-53; and the pair's own 2^-48 of the output.  A lost diagonal of digit
products would stand out by a factor of 2^8.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <vector>
#include "kernels.h"
using namespace ofdft;
extern "C" int run(const int *grid, int axis, int kind, double scale, const float *in, float *out)
{
    GridInfo g{};
    g.nx = grid[0]; g.ny = grid[1]; g.nz = grid[2];
    g.K = g.nz / 2 + 1;
    g.N = (long long)g.nx * g.ny * g.nz;
    const int n = grid[axis];
    if (!tline_supported(n)) return 1;
    std::vector<uint16_t> img(tline_matrix_bytes(n) / 2);
    TlMat m;
    m.mexp = kind == 0 ? tline_derivative_matrix(n, scale, img.data()) : tline_fourier_matrix(n, kind == 2, img.data());
    void *mat = nullptr, *buf = nullptr;
    if (cudaMalloc(&mat, img.size() * 2) != cudaSuccess || cudaMalloc(&buf, 16 * (size_t)g.N) != cudaSuccess) return 2;
    m.img = mat;
    float2 *a = (float2 *)buf, *b = a + g.N;
    cudaMemcpy(mat, img.data(), img.size() * 2, cudaMemcpyHostToDevice);
    cudaMemcpy(a, in, 8 * (size_t)g.N, cudaMemcpyHostToDevice);
    cudaDeviceSynchronize();
    if (tline_smem_limits() != cudaSuccess) return 3;
    const TlPass p = {kind == 0 ? TlPass::kDerivative : kind == 1 ? TlPass::kForward : TlPass::kInverse, axis, &m, a, b};
    launch_tline(g, 1, &p, 0);
    cudaMemcpy(out, b, 8 * (size_t)g.N, cudaMemcpyDeviceToHost);
    const int bad = cudaGetLastError() == cudaSuccess ? 0 : 4;
    cudaFree(mat);
    cudaFree(buf);
    return bad;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import __graft_entry__
    __graft_entry__.build()
    d = tmp_path_factory.mktemp("tl")
    src, so = d / "tl.cu", d / "tl.so"
    src.write_text(SRC)
    pkg = os.path.join(ROOT, "paper_1406_0835_gb300")
    libdir = os.path.join(pkg, "_build")
    subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                           "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I" + os.path.join(pkg, "csrc"),
                           str(src), "-o", str(so), "-L" + libdir, "-lofdft", "-lcudart",
                           "-Xlinker", "-rpath=" + libdir])
    lib = ctypes.CDLL(str(so))
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p]
    return lib


def fourier(n):
    """The orthonormal real Fourier matrix: even frequencies first (0; 2 cos, 2 sin; ...), then the odd ones."""
    h = n // 2
    rows = [(0, False)] + [(2 * ((i + 1) // 2), i % 2 == 0) for i in range(1, h)]
    rows += [(2 * (i // 2) + 1, i % 2 == 1) for i in range(h)]
    pi = np.longdouble("3.14159265358979323846264338327950288")
    out = np.empty((n, n), dtype=np.longdouble)
    for a, (k, sine) in enumerate(rows):
        x = 2 * pi * ((k * np.arange(n)) % n) / n
        norm = np.sqrt(np.longdouble(1 if k in (0, h) else 2) / n)
        out[a] = norm * (np.sin(x) if sine else np.cos(x))
    return out


def derivative(n, scale):
    pi = np.longdouble("3.14159265358979323846264338327950288")
    m = (np.arange(n)[:, None] - np.arange(n)[None, :]) % n
    x = pi * m.astype(np.longdouble) / n
    with np.errstate(all="ignore"):
        cot = np.where((m == 0) | (2 * m == n), np.longdouble(0), np.cos(x) / np.where(m == 0, np.longdouble(1), np.sin(x)))
    return np.longdouble(scale) / 2 * np.where(m % 2 == 1, -cot, cot)


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", [8, 10, 18, 32, 50, 64, 90, 128, 144])
def test_one_transform(run, n, axis, kind):
    grid = [8, 10, 12]
    grid[axis] = n
    rng = np.random.default_rng(1000 * n + 10 * axis + kind)
    x = rng.standard_normal(grid) * 10.0 ** rng.uniform(-6, 6, [1 if a == axis else g for a, g in enumerate(grid)])
    hi = x.astype(np.float32)
    lo = (x - hi).astype(np.float32)
    pairs = np.stack([hi, lo], axis=-1)
    got = np.empty_like(pairs)
    sizes = np.array(grid, dtype=np.int32)
    assert run.run(sizes.ctypes.data, axis, kind, 0.7, pairs.ctypes.data, got.ctypes.data) == 0
    M = derivative(n, 0.7) if kind == 0 else (fourier(n) if kind == 1 else fourier(n).T)
    xl = np.moveaxis(np.longdouble(hi) + np.longdouble(lo), axis, -1)
    want = xl @ M.T
    out = np.moveaxis(np.longdouble(got[..., 0]) + np.longdouble(got[..., 1]), axis, -1)
    top = np.abs(xl).max(axis=-1, keepdims=True) * np.abs(M).max()
    one = np.sqrt((top * (np.sqrt(6.0 * n) * 2.0 ** -52.6 + np.sqrt(n) * 2.0 ** -53)) ** 2 + (2.0 ** -48 * want) ** 2)
    assert np.sqrt(np.mean(((out - want) / one) ** 2)) < 2.0
