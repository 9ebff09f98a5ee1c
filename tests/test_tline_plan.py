"""CPU: which axes and chains of a double-float set run on the tensor cores
(tline_plan), called from the library through a small host program.  A GGA
set takes the real-basis form only with all three derivative matrices: a grid
spacing whose matrix leaves the exponent range keeps that axis, and with it
the Hartree chain, on the FFT passes, and axes of one length never share a
matrix that is not there.  Laying out matrices takes no host memory (the
allocation-free entry point does it on its first call).  The GPU case evaluates such a cell."""
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1406_0835_gb300", "csrc")
LIBDIR = os.path.join(ROOT, "paper_1406_0835_gb300", "_build")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>
#include "kernels.h"
using namespace ofdft;
static long long news = 0;             // also counts the library's
void *operator new(size_t n)
{
    ++news;
    if (void *p = malloc(n)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
int main(int, char **v)
{
    GridInfo g{};
    g.nx = atoi(v[1]); g.ny = atoi(v[2]); g.nz = atoi(v[3]);
    g.K = g.nz / 2 + 1;
    g.N = (long long)g.nx * g.ny * g.nz;
    g.Lx = atof(v[4]); g.Ly = atof(v[5]); g.Lz = atof(v[6]);
    g.omega = g.Lx * g.Ly * g.Lz;
    g.dd = 1;
    grid_reciprocal(g);
    const TlPlan p = tline_plan(g, atoi(v[7]) != 0);
    const int n3[3] = {g.nx, g.ny, g.nz};
    printf("%d %d %d %d", p.der[0], p.der[1], p.der[2], p.real_basis);
    for (int a = 0; a < 3; ++a) {      // the exponent the matrix really gets
        int e = 999;
        if (tline_supported(n3[a])) {
            std::vector<uint16_t> img(tline_matrix_bytes(n3[a]) / 2);
            const long long before = news;
            e = tline_derivative_matrix(n3[a], g.ds[a] * n3[a], img.data());
            for (int inv = 0; inv < 2; ++inv) tline_fourier_matrix(n3[a], inv, img.data());
            news -= before;
        } else {
            news = 0;
        }
        printf(" %d %lld", e, news);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    import __graft_entry__
    __graft_entry__.build()
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cpp", d / "plan"
    src.write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I" + CSRC, "-I/usr/local/cuda/include", str(src), "-o", str(exe),
                           "-L" + LIBDIR, "-lofdft", "-Wl,-rpath," + LIBDIR, "-Wl,-rpath,/usr/local/cuda/lib64"])

    def run(grid, L, gga):
        out = subprocess.check_output([str(exe)] + [str(x) for x in (*grid, *L, int(gga))]).split()
        return [x == b"1" for x in out[:3]], out[3] == b"1", [int(x) for x in out[4::2]], [int(x) for x in out[5::2]]
    return run


@pytest.mark.parametrize("grid", [(16, 16, 16), (8, 16, 96), (144, 10, 16), (96, 150, 12)])
@pytest.mark.parametrize("spacing", [(0.25, 0.25, 0.25), (2.0e4, 2.0e4, 2.0e4), (0.25, 2.0e4, 0.25), (1.0e-6, 300.0, 1.5e4),
                                     (1.0e5, 0.3, 0.3), (1.0e-40, 1.0, 1.0)])
def test_a_set_takes_the_form_its_matrices_allow(plan, grid, spacing):
    L = [n * s for n, s in zip(grid, spacing)]
    der, real, mexp, news = plan(grid, L, True)
    assert der == [-60 <= e <= 68 for e in mexp]
    assert real == all(der)
    assert news == [0, 0, 0]
    der, real, _, _ = plan(grid, L, False)
    assert der == [False] * 3
    assert real == all(n <= 144 for n in grid)


@pytest.mark.gpu
def test_a_cell_of_large_spacings_is_computed():
    """16^3 points 20,000 bohr apart, VT84F (bars as the other parity tests)."""
    import oracle as O
    from paper_1406_0835_gb300 import ofdft
    grid, L = (16, 16, 16), [3.2e5] * 3
    ions = np.random.default_rng(5).random((30, 3)) * L
    so = O.System(L, grid, ions, np.ones(30), 1.0e5, "vt84f")
    phi = so.uniform_phi() * (1.0 + 0.1 * np.random.default_rng(6).standard_normal(grid))
    ev = O.evaluate(so, phi)
    with ofdft.Context(L, grid, ions, np.ones(30), 1.0e5, "vt84f") as ctx:
        E, v = ctx.energy_potential(phi)
    for k in ("F_tot", "F_s", "F_xc", "E_H"):
        assert abs(E[k] - ev[k]) <= 1e-10 * abs(ev["F_tot"]), (k, E[k], ev[k])
    assert np.max(np.abs(v - ev["v"])) <= 1e-9 * np.max(np.abs(ev["v"]))
