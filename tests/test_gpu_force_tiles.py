"""GPU parity of the tensor-core local forces at sizes that the dispatch rule
gives them (points times ions, rounded up to 32, from 4e6), with the launch
count as the witness that they took the call: one ion, one ragged group of
64, two groups, z edges below one block of 64 coefficients, across it, and
ending inside a chunk of 16, y edges that are no multiple of the 32-row tile,
odd half lengths.  Densities rough enough that every Nyquist line and corner
carries weight.  Bar as the other force parity test: 1e-10 Ha/bohr (N products
of 53-bit digits with pairs, 2^-44 of about 1 Ha/bohr, and the ion-ion sums)."""
import numpy as np
import pytest

import oracle as O
from paper_1406_0835_gb300 import inputs, ofdft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("grid,nat,lpp", [((50, 50, 54), 1, "gauss"), ((40, 54, 90), 33, "gauss"), ((54, 60, 50), 63, "ha"),
                                          ((60, 72, 30), 64, "gauss"), ((144, 144, 10), 40, "ha"), ((36, 40, 144), 17, "gauss"),
                                          ((48, 50, 64), 65, "ha"), ((8, 90, 72), 100, "gauss")])
def test_forces_match_the_oracle(grid, nat, lpp):
    assert np.prod(grid) * (-(-nat // 32) * 32) >= 4e6
    rng = np.random.default_rng(nat + sum(grid))
    L = np.array([7.0, 8.0, 9.0])
    ions = inputs.random_positions(nat, 8.0, nat, 4.0 / nat ** (1.0 / 3.0)) / 8.0 * L
    so = O.System(list(L), grid, ions, np.ones(nat), 5.0e4, "sga", lpp=lpp)
    phi = so.uniform_phi() * (1.0 + 0.1 * rng.standard_normal(grid))
    phi *= np.sqrt(nat / (np.sum(phi * phi) * np.prod(L) / np.prod(grid)))
    F_o = O.forces(so, O.evaluate(so, phi))
    with ofdft.Context(list(L), grid, ions, np.ones(nat), 5.0e4, "sga", lpp=lpp) as ctx:
        ctx.set_phi(phi)
        before = ctx.kernel_launches()
        F, _ = ctx.forces()
        n = ctx.kernel_launches() - before
        ctx.energy_potential(None, want_v=False)
        evaluation = ctx.kernel_launches() - before - n
    # an evaluation, n(G) in three, then coefficients, phases, forces, their sums (the other form: three)
    assert n == evaluation + 3 + 4
    assert np.max(np.abs(F - F_o)) <= 1e-10
