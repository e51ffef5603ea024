"""Rate coefficients when kT is far above the last computed energy: the integral is then mostly the power-law tail
(U/U_K)^p, whose incomplete gamma function Gamma(2 + p, U_K/kT) the closed form has to give over p in [-1, 0]
for U_K/kT from 10 down to 1e-12, against the oracle (1e-12 relative: the library's documented 1e-13, the
oracle's adaptive quadrature at 1e-13, the power of kT and its logarithm of a few 1e-14)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x", [10.0, 1.0, 0.3, 0.1, 0.0999, 0.03, 1e-2, 1e-4, 1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("p", [-1.0, -0.95, -0.5, -0.05, 0.0])
def test_tail(x, p):
    from oracle import rates as R

    import paper_2312_02322_gb300.api as mq

    U = 1e-4 * np.array([1.0, 2.0, 4.0])
    # sigma = s U^p at the three energies (p = -1: a little steeper, so that the exponent is clipped)
    L = 3
    E = np.array([0.0, 0.5 * U[0], 2.5 * U[0]])
    g = np.array([1.0, 3.0, 5.0])
    s = np.array([[1.0, 2.0, 0.5], [0.7, 3.0, 1.1], [0.2, 0.9, 4.0]])
    slope = p if p > -1.0 else -1.02
    sig = s[None] * (U[:, None, None] / U[0]) ** slope
    kT = np.array([U[-1] / x])
    _, rate = mq.rate_coefficients(sig, U, E, g, 3000.0, kT)
    ref = R.rates(sig, U, E, g, 3000.0, kT)
    assert rate.shape == (1, L, L) and np.all(ref > 0.0)
    assert np.max(np.abs(rate / ref - 1.0)) < 1e-12
