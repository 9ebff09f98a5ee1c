"""CPU: rms errors of the double-float quotient, reciprocal and square root
(host branches).  With binary32 divisions and a double-float remainder they
are 0.61, 0.48 and 0.32 u^2 (u^2 = 2^-48) over operands uniform in an octave;
the forms without divisions may not be further off than 10 % above that."""
import numpy as np
import pytest

from paper_1406_0835_gb300 import ofdft


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("op,bar", [("div", 0.67), ("recip", 0.53), ("sqrt", 0.35)])
def test_rms(op, bar):
    rng = np.random.default_rng(4)

    def dd(x):
        hi = np.float32(x).astype(np.float64)
        return hi + np.float32(x - hi).astype(np.float64)
    n = 200000
    x, y = dd(rng.uniform(1.0, 2.0, n)), dd(rng.uniform(1.0, 2.0, n))
    if op == "sqrt":
        x = dd(rng.uniform(1.0, 4.0, n))
        got, want = ofdft.ofdft_ffmath_eval("sqrt", x), np.sqrt(np.longdouble(x))
    else:
        if op == "recip":
            x = np.ones(n)
        got, want = ofdft.ofdft_ffmath_eval("div", x, y), np.longdouble(x) / np.longdouble(y)
    err = (np.longdouble(got) - want) / want * 2.0 ** 48
    assert np.sqrt(np.mean(err ** 2)) < bar
