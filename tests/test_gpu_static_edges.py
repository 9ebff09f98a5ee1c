"""The allocation-free entry point on every edge it takes (its transform
matrices are laid out per edge, with unit spacing) in uneven cells, ftTF and
GGA, against the oracle.  Bars as the other parity tests: energies 1e-10 of
F_tot, the potential 1e-9 of its maximum."""
import numpy as np
import pytest

import oracle as O
from paper_1406_0835_gb300 import inputs, ofdft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("functional", ["fttf", "vt84f"])
@pytest.mark.parametrize("grid", [(8, 8, 8), (10, 12, 16), (18, 20, 24), (30, 32, 8), (36, 40, 10), (12, 48, 50), (54, 8, 60),
                                  (64, 8, 64)])
def test_every_edge(grid, functional):
    import torch
    rng = np.random.default_rng(sum(grid))
    L = np.array([4.0, 5.5, 7.0])
    ions = inputs.random_positions(9, 4.0, 11, 0.8) / 4.0 * L
    so = O.System(list(L), grid, ions, np.ones(9), 8.0e4, functional)
    phi = so.uniform_phi() * (1.0 + 0.1 * rng.standard_normal(grid))
    ev = O.evaluate(so, phi)
    p = torch.as_tensor(phi.reshape(-1), device="cuda")
    v = torch.empty_like(p)
    E = ofdft.ofdft_energy_potential_static(np.diag(L), grid, ions, np.ones(9), 8.0e4, functional, p.data_ptr(), v.data_ptr())
    for k in ("F_tot", "F_s", "F_xc", "E_H", "E_loc"):
        assert abs(E[k] - ev[k]) <= 1e-10 * abs(ev["F_tot"]), (k, E[k], ev[k])
    assert np.max(np.abs(v.cpu().numpy().reshape(grid) - ev["v"])) <= 1e-9 * np.max(np.abs(ev["v"]))
