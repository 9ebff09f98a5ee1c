"""The allocation-free entry point's ion-ion energy (Ewald sums on the
device) against the context path's: one ion, two, the largest count, ions
outside the cell and exactly half a cell apart (a tie of the minimum image),
uneven cells, and a cell so long that the sums stay on the host.  Both sum
the same converged series in binary64, so they agree to 1e-12 of the sum of
the terms' magnitudes."""
import numpy as np
import pytest

from paper_1406_0835_gb300 import ofdft

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nat,L,shift", [(1, (4.0, 4.0, 4.0), 0.0), (2, (4.0, 5.0, 6.0), 0.0), (7, (3.0, 9.0, 4.5), 1.0e4),
                                         (64, (8.0, 8.0, 8.0), -3.0), (33, (5.0, 5.0, 40.0), 0.0),
                                         (5, (2.0, 2.0, 400.0), 0.0)])
def test_ion_energy(nat, L, shift):
    import torch
    rng = np.random.default_rng(nat)
    L = np.array(L)
    ions = rng.random((nat, 3)) * L + shift * L
    if nat == 2:
        ions = np.array([[0.25, 0.5, 0.75], [0.75, 0.0, 0.25]]) * L
    Z = 1.0 + (np.arange(nat) % 3)
    grid = (8, 10, 12)
    N = int(np.prod(grid))
    phi = torch.full((N,), float(np.sqrt(Z.sum() / L.prod())), dtype=torch.float64, device="cuda")
    v = torch.empty_like(phi)
    E = ofdft.ofdft_energy_potential_static(np.diag(L), grid, ions, Z, 1.0e5, "fttf", phi.data_ptr(), v.data_ptr())
    with ofdft.Context(L, grid, ions, Z, 1.0e5, "fttf") as ctx:
        ref, _ = ctx.energy_potential(None, want_v=False)
    scale = float((Z * Z).sum()) / L.min() + abs(ref["E_ion"])
    assert abs(E["E_ion"] - ref["E_ion"]) <= 1e-12 * scale
    E2 = ofdft.ofdft_energy_potential_static(np.diag(L), grid, ions, Z, 1.0e5, "fttf", phi.data_ptr(), v.data_ptr())
    assert E2["E_ion"] == E["E_ion"]          # the sums do not depend on scheduling
