"""GPU: the tensor-core force sums by themselves (launch_force_tc on given
coefficients, corners zero) against the sums in extended precision, on rows
whose largest coefficient is that of frequency 0 along z, where the z force
has no term: what the others weigh must not be rounded to its size.

Bar, per ion and axis: six standard deviations of independent roundings.  A
coefficient is a pair, 2^-49 of itself, each product and sum of pairs a few
2^-48 of its size (8 allowed, of the root of the terms' squares); a row's
digits round to 2^-60 of twice its largest value, the phases to 2^-55 (f_c' of
the block's highest frequency times 4/7; frequency 0's are exact), uniformly."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "kernels.h"
using namespace ofdft;
// coef: nx ny nz pairs; F: nat x 3
extern "C" int run(const int *grid, const double *L, int nat, const double *R, const float *coef, double *F)
{
    GridInfo g{};
    g.nx = grid[0]; g.ny = grid[1]; g.nz = grid[2];
    g.K = g.nz / 2 + 1;
    g.N = (long long)g.nx * g.ny * g.nz;
    g.NH = (long long)g.nx * g.ny * g.K;
    g.Lx = L[0]; g.Ly = L[1]; g.Lz = L[2];
    g.omega = L[0] * L[1] * L[2];
    g.dV = g.omega / (double)g.N;
    g.rc = 0.25;
    g.dd = 1;
    grid_reciprocal(g);
    if (!force_tc_takes(g, nat) || force_tc_smem_limits() != cudaSuccess) return 1;
    const size_t np = (size_t)nat * (g.nx + g.ny + g.K), chunks = (size_t)force_tc_chunks(g, nat);
    double *Rd, *Z, *part, *Fd;
    double2 *ph, *nG;
    float2 *c;
    void *scratch;
    if (cudaMalloc(&Rd, 24 * (size_t)nat) || cudaMalloc(&Z, 8 * (size_t)nat) || cudaMalloc(&part, 24 * nat * chunks) ||
        cudaMalloc(&Fd, 24 * (size_t)nat) || cudaMalloc(&ph, 16 * np) || cudaMalloc(&nG, 16 * (size_t)g.NH) ||
        cudaMalloc(&c, 8 * (size_t)g.N) || cudaMalloc(&scratch, force_tc_bytes(g, nat)))
        return 2;
    cudaMemcpy(Rd, R, 24 * (size_t)nat, cudaMemcpyHostToDevice);
    cudaMemcpy(c, coef, 8 * (size_t)g.N, cudaMemcpyHostToDevice);
    cudaMemset(nG, 0, 16 * (size_t)g.NH);
    launch_fill<double>(nat, Z, 1.0, 0);
    double2 *px = ph, *py = px + (size_t)nat * g.nx, *pz = py + (size_t)nat * g.ny;
    launch_phases(g, nat, Rd, px, py, pz, nullptr, 0);
    const int n = launch_force_tc(g, nat, Z, px, py, pz, nG, c, scratch, part, 0);
    launch_force_reduce(nat, n, part, Fd, 0, 0);
    cudaMemcpy(F, Fd, 24 * (size_t)nat, cudaMemcpyDeviceToHost);
    const int bad = cudaGetLastError() == cudaSuccess ? 0 : 3;
    for (void *p : {(void *)Rd, (void *)Z, (void *)part, (void *)Fd, (void *)ph, (void *)nG, (void *)c, scratch}) cudaFree(p);
    return bad;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import __graft_entry__
    __graft_entry__.build()
    d = tmp_path_factory.mktemp("fc")
    src, so = d / "fc.cu", d / "fc.so"
    src.write_text(SRC)
    pkg = os.path.join(ROOT, "paper_1406_0835_gb300")
    libdir = os.path.join(pkg, "_build")
    subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                           "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I" + os.path.join(pkg, "csrc"),
                           str(src), "-o", str(so), "-L" + libdir, "-lofdft", "-lcudart",
                           "-Xlinker", "-rpath=" + libdir])
    lib = ctypes.CDLL(str(so))
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int] + [ctypes.c_void_p] * 3
    return lib


def phases(n, L, r):
    """Cosine (0 and odd index) or sine of frequency (c + 1) // 2 at r, and its derivative per phase."""
    pi = np.longdouble("3.14159265358979323846264338327950288")
    c = np.arange(n)
    k = (c + 1) // 2
    x = np.longdouble(2) * pi * k * (np.longdouble(r) / np.longdouble(L))
    sine = (c > 0) & (c % 2 == 0)
    return np.where(sine, np.sin(x), np.cos(x)), k * np.where(sine, np.cos(x), -np.sin(x))


@pytest.mark.parametrize("grid,nat", [((64, 64, 64), 32), ((30, 36, 128), 33), ((50, 48, 90), 20)])
def test_small_terms_beside_a_large_constant(run, grid, nat):
    nx, ny, nz = grid
    rng = np.random.default_rng(nz)
    L = np.array([8.0, 7.0, 9.0])
    R = rng.random((nat, 3)) * L
    c = np.arange(nz)
    g = rng.standard_normal(grid) * np.where(c == 0, 1.0, 2.0 ** -14 * np.exp(-0.05 * c))
    hi = g.astype(np.float32)
    lo = (g - hi).astype(np.float32)
    pairs = np.ascontiguousarray(np.stack([hi, lo], axis=-1))
    F = np.empty((nat, 3))
    sizes = np.array(grid, dtype=np.int32)
    assert run.run(sizes.ctypes.data, L.ctypes.data, nat, R.ctypes.data, pairs.ctypes.data, F.ctypes.data) == 0
    G = np.longdouble(hi) + np.longdouble(lo)
    b = 2.0 * np.pi / L
    top = np.abs(g).max(axis=2)
    for i in range(nat):
        (fx, dx), (fy, dy), (fz, dz) = (phases(n, L[a], R[i, a]) for a, n in enumerate(grid))
        T, Tp = G @ fz, G @ dz
        want = np.array([dx @ T @ fy, fx @ T @ dy, fx @ Tp @ fy])
        for a, (u, v, w) in enumerate([(dx, fy, fz), (fx, dy, fz), (fx, fy, dz)]):
            uv = np.outer(np.abs(u), np.abs(v)).astype(np.float64)
            terms = np.sqrt(np.einsum("xy,xyz,z->", uv ** 2, g ** 2, w.astype(np.float64) ** 2))
            w2 = np.sqrt(np.sum(w.astype(np.float64) ** 2))
            digits = np.sqrt(np.sum((uv * top) ** 2)) * w2 * 2.0 ** -59 / np.sqrt(12.0)
            scale = nz / 2.0 * 4.0 / 7.0 if a == 2 else 1.0
            phase = np.sqrt(np.einsum("xy,xyz->", uv ** 2, g[:, :, 1:] ** 2)) * 2.0 ** -54 / np.sqrt(12.0) * scale
            bar = 6.0 * b[a] * np.sqrt((8.0 * 2.0 ** -48 * terms) ** 2 + digits ** 2 + phase ** 2)
            assert abs(float(np.longdouble(F[i, a]) - np.longdouble(b[a]) * want[a])) <= bar, (i, a)
