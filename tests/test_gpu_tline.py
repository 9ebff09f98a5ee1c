"""GPU parity of the tensor-core transforms (kernels_tline.cu: derivatives,
and the Hartree chain in the real Fourier basis) at the
sizes where their tiling can go wrong: the smallest edges, odd half lengths,
edges whose halves are no multiple of the padding, one, two and three column
chunks, the largest edge they take (144) and the first beyond it (150, which
keeps the double-float transforms), line counts that leave a ragged tile,
and a sheared cell.  The GGA energy and potential against the oracle.

Bars as the other parity tests: energies 1e-10 of F_tot, the potential 1e-9
of its maximum.  A density with a non-finite value is refused, as by the
other evaluation paths.
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


def check(grid, cell=None, functional="vt84f"):
    cfg = inputs.config_single_point()
    L = np.array(cfg["L"])
    ions = cfg["ions"] if cell is None else (cfg["ions"] / L) @ cell
    kw = {} if cell is None else {"cell": cell}
    so = O.System(None if cell is not None else cfg["L"], grid, ions, cfg["Z"], cfg["T"], functional, **kw)
    rng = np.random.default_rng(sum(grid))
    phi = so.uniform_phi() * (1.0 + 0.1 * rng.standard_normal(grid))
    ev = O.evaluate(so, phi)
    with ofdft.Context(None if cell is not None else cfg["L"], grid, ions, cfg["Z"], cfg["T"], functional, **kw) as ctx:
        E, v = ctx.energy_potential(phi)
    for k in ("F_tot", "F_s", "F_xc", "E_H"):
        assert abs(E[k] - ev[k]) <= 1e-10 * abs(ev["F_tot"]), (k, E[k], ev[k])
    assert np.max(np.abs(v - ev["v"])) <= 1e-9 * np.max(np.abs(ev["v"]))


@pytest.mark.parametrize("grid", [(8, 8, 8), (10, 18, 30), (50, 54, 10), (12, 128, 16), (144, 8, 10), (8, 10, 144),
                                  (150, 16, 12), (12, 10, 150), (20, 36, 90), (96, 40, 8)])
def test_evaluation_at_the_edges_of_the_tiling(grid):
    check(grid)


@pytest.mark.parametrize("grid", [(60, 54, 50), (144, 36, 40)])
def test_fttf_grids_large_enough_for_the_real_basis(grid):
    check(grid, functional="fttf")


def test_heine_abarenkov_weights_in_the_real_basis():
    """Pressure weights and v_ext of Eq. (E4A), odd half lengths on two axes."""
    cfg = inputs.config_single_point()
    grid = (18, 20, 30)
    so = O.System(cfg["L"], grid, cfg["ions"], cfg["Z"], cfg["T"], "sga", lpp="ha")
    rng = np.random.default_rng(3)
    phi = so.uniform_phi() * (1.0 + 0.1 * rng.standard_normal(grid))
    ev = O.evaluate(so, phi)
    with ofdft.Context(cfg["L"], grid, cfg["ions"], cfg["Z"], cfg["T"], "sga", lpp="ha") as ctx:
        E, v = ctx.energy_potential(phi)
    for k in ("F_tot", "E_H", "E_loc"):
        assert abs(E[k] - ev[k]) <= 1e-10 * abs(ev["F_tot"]), k
    for k in ("P", "P_H", "P_loc"):
        assert abs(E[k] - ev[k]) <= 1e-9 * abs(ev["P"]), k
    assert np.max(np.abs(v - ev["v"])) <= 1e-9 * np.max(np.abs(ev["v"]))


def test_sheared_cell():
    L = np.array(inputs.config_single_point()["L"])
    check((20, 54, 36), np.diag(L) + np.array([[0.0, 0.0, 0.0], [0.45, 0.0, 0.0], [-0.3, 0.55, 0.0]]))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_density_is_refused(bad):
    cfg = inputs.config_single_point()
    phi = np.full((16, 18, 20), 0.3)
    phi[3, 4, 5] = bad
    with ofdft.Context(cfg["L"], phi.shape, cfg["ions"], cfg["Z"], cfg["T"], "vt84f") as ctx:
        with pytest.raises(ofdft.OfdftError) as e:
            ctx.energy_potential(phi)
        assert e.value.status == -4


@pytest.mark.parametrize("grid", [(8, 16, 16), (10, 12, 16), (12, 10, 18), (36, 8, 10)])
def test_fttf_grids_on_both_sides_of_the_rule(grid):
    """2048 points and more take the real basis; 1920 keep the FFT passes."""
    check(grid, functional="fttf")


@pytest.mark.parametrize("functional,lpp", [("fttf", "gauss"), ("vt84f", "ha")])
@pytest.mark.parametrize("grid", [(8, 16, 16), (10, 18, 30), (36, 20, 8), (12, 50, 18)])
def test_real_basis_in_sheared_cells(grid, functional, lpp):
    """Every Nyquist plane, line and corner carries weight (rough density) and
    the cell has no right angle."""
    cfg = inputs.config_single_point()
    L = np.array(cfg["L"])
    cell = np.diag(L) + np.array([[0.0, 0.3, -0.2], [0.8, 0.0, 0.4], [-0.5, 0.9, 0.0]])
    ions = (cfg["ions"] / L) @ cell
    so = O.System(None, grid, ions, cfg["Z"], cfg["T"], functional, cell=cell, lpp=lpp)
    phi = so.uniform_phi() * (1.0 + 0.1 * np.random.default_rng(sum(grid)).standard_normal(grid))
    ev = O.evaluate(so, phi)
    with ofdft.Context(None, grid, ions, cfg["Z"], cfg["T"], functional, cell=cell, lpp=lpp) as ctx:
        E, v = ctx.energy_potential(phi)
    for k in ("F_tot", "F_s", "F_xc", "E_H", "E_loc"):
        assert abs(E[k] - ev[k]) <= 1e-10 * abs(ev["F_tot"]), (k, E[k], ev[k])
    for k in ("P", "P_loc"):
        assert abs(E[k] - ev[k]) <= 1e-9 * abs(ev["P"]), (k, E[k], ev[k])
    assert np.max(np.abs(v - ev["v"])) <= 1e-9 * np.max(np.abs(ev["v"]))
