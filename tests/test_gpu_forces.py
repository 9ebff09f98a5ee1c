"""GPU parity of the tensor-core local forces (kernels_force.cu) at the sizes
where their tiling can go wrong: the fewest ions it takes, one and two groups
of 64 ions with a ragged last one, z edges below, at and above one block of
64 coefficients, y edges that are no multiple of the 32-row tile, odd half
lengths, both ion models.  The densities are rough, so that every Nyquist
line and corner carries weight.

Bar: each force is a sum of N products of 53-bit digits with pairs, so within
2^-44 of the sum of the terms' magnitudes, about 1 Ha/bohr here; the ion-ion
force beside it, up to 10 Ha/bohr, is a binary64 sum of the same accuracy as
the oracle's (1e-13 of it).  1e-10 Ha/bohr leaves a factor of 50 to both.
"""
import numpy as np
import pytest

import oracle as O
from paper_1406_0835_gb300 import inputs, ofdft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("lpp", ["gaussian", "ha"])
@pytest.mark.parametrize("grid,nat", [((8, 8, 8), 16), ((10, 18, 30), 65), ((8, 30, 64), 17), ((12, 32, 72), 64),
                                      ((16, 36, 128), 130), ((30, 36, 10), 40), ((8, 10, 144), 63)])
def test_forces_match_the_oracle(grid, nat, lpp):
    rng = np.random.default_rng(nat + sum(grid))
    L = np.array([7.0, 8.0, 9.0])
    ions = inputs.random_positions(nat, 8.0, nat, 4.0 / nat ** (1.0 / 3.0)) / 8.0 * L
    Z = np.ones(nat)
    kw = {} if lpp == "gaussian" else {"lpp": "ha"}
    so = O.System(list(L), grid, ions, Z, 5.0e4, "sga", **kw)
    phi = so.uniform_phi() * (1.0 + 0.1 * rng.standard_normal(grid))
    phi *= np.sqrt(nat / (np.sum(phi * phi) * np.prod(L) / np.prod(grid)))
    F_o = O.forces(so, O.evaluate(so, phi))
    with ofdft.Context(list(L), grid, ions, Z, 5.0e4, "sga", **kw) as ctx:
        ctx.set_phi(phi)
        F, _ = ctx.forces()
    assert np.max(np.abs(F - F_o)) <= 1e-10
