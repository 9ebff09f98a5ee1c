"""GPU: the work of forces and of ofdft_autotune on sets in the real-basis
form.  n(G) for ftTF forces falls out of the FFT form's own x pass, so that
call makes no evaluation of the other form beside three passes for n(G);
autotune times the FFT passes that the forces and the stress of a real-basis
set still take.  Counted in kernel launches; forces and energies agree with
an untuned context to rounding (1e-12 of their scale)."""
import numpy as np
import pytest

from paper_1406_0835_gb300 import inputs, ofdft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def context(functional, grid):
    d = inputs.hydrogen(8, 1.0, 1.0e5, grid, seed=7, functional=functional)
    ctx = ofdft.Context(d["L"], grid, d["ions"], d["Z"], d["T"], functional)
    rng = np.random.default_rng(sum(grid))
    ctx.set_phi(np.sqrt(8.0 / np.prod(d["L"])) * (1.0 + 0.1 * rng.standard_normal(grid)))
    return ctx


def launches(ctx, call):
    before = ctx.kernel_launches()
    out = call()
    return ctx.kernel_launches() - before, out


@pytest.mark.parametrize("grid", [(8, 16, 16), (24, 30, 32), (144, 10, 12)])
def test_fttf_forces_take_n_of_G_from_the_evaluation(grid):
    with context("fttf", grid) as ctx:
        n, (F, P) = launches(ctx, ctx.forces)
        assert n == 6 + 3                   # z, y, x, y, z, sums; weights, forces, their sums
        n, (E, _) = launches(ctx, lambda: ctx.energy_potential(None, want_v=False))
        assert n == 10                      # the real-basis form
    assert abs(P - E["P"]) <= 1e-12 * (abs(E["P_s"]) + abs(E["P_H"]) + abs(E["P_loc"]) + abs(E["P_ion"]))


# (grids of their own: the shapes found are kept per grid for the process)
@pytest.mark.parametrize("functional,grid", [("fttf", (30, 24, 36)), ("vt84f", (36, 24, 30))])
def test_autotune_times_the_passes_that_are_left(functional, grid):
    with context(functional, grid) as a, context(functional, grid) as b:
        n, _ = launches(a, lambda: a.autotune(reps=2))
        assert n > 0
        E, Ea = b.energy_potential(None, want_v=False)[0], a.energy_potential(None, want_v=False)[0]
        assert E == Ea                      # real-basis evaluations have one shape
        (F, _), (Fa, _) = b.forces(), a.forces()
        assert np.max(np.abs(F - Fa)) <= 1e-12 * np.max(np.abs(F))
        a.set_phi()
        b.set_phi()
        assert a.minimize(gtol=1e-6)[0]["F_tot"] == b.minimize(gtol=1e-6)[0]["F_tot"]
