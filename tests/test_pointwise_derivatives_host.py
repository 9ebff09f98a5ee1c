"""CPU: df/dn of the double-float functional where the temperature
polynomials' ends meet (t at the edges of the refined panels, where their
highest degrees weigh most in the t-derivatives) and s^2 is large, so that
df/dn hangs on the derivatives of A and B.

Bar: df/dn is a sum of four products of about ten pair operations, each
within 5 2^-48 of its operands, so within 50 2^-48 = 1.8e-13 of the terms'
size (|df/dn| + (|f| + |T s|) / n, as in the other pointwise tests)."""
import numpy as np
import pytest

import oracle as O
from paper_1406_0835_gb300 import ofdft

OF_CS = 1.0 / (4.0 * (3.0 * np.pi ** 2) ** (2.0 / 3.0))


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("fn", ["sga", "vt84f", "kst2", "tw"])
@pytest.mark.parametrize("T_kelvin", [3.0e4, 1.0e6])
def test_derivatives_at_the_panels_edges(fn, T_kelvin):
    rng = np.random.default_rng(12)
    edge = 2.0 ** np.arange(-4, 6)[:, None] * (1.0 + np.arange(16)[None, :] / 16.0)
    t = np.concatenate([edge.ravel() * (1.0 + s * rng.uniform(1e-6, 1e-3, (20, edge.size))).ravel().reshape(20, -1)
                        for s in (-1.0, 1.0)]).ravel()
    n = (2.0 * T_kelvin * O.KB_HA_PER_K / t) ** 1.5 / (3.0 * np.pi ** 2)
    s2 = 10.0 ** rng.uniform(1.3, 3.0, n.size)
    g2 = s2 * n ** (8.0 / 3.0) / OF_CS
    a, used = ofdft.ofdft_pointwise_eval(fn, True, T_kelvin, n, g2, "f32x2")
    b, _ = ofdft.ofdft_pointwise_eval(fn, True, T_kelvin, n, g2, "f64")
    assert used == n.size
    err = np.abs(a[:, 2] - b[:, 2]) / (np.abs(b[:, 2]) + (np.abs(b[:, 0]) + np.abs(b[:, 1])) / n)
    assert np.max(err) < 50.0 * 2.0 ** -48
