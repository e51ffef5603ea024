"""The closed form of the rate integrals where it can go wrong: thresholds on, between, below and above the
knots, two to 32 energies, level counts around the 16 x 8 pair tiles, z = (U - u0)/kT on both sides of the
incomplete gamma functions' switch, against the oracle's adaptive quadrature (relative 1e-10)."""
import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mq():
    import torch

    assert torch.cuda.is_available()
    import paper_2312_02322_gb300.api as api

    return api


@pytest.mark.parametrize("K,L", [(2, 9), (3, 17), (10, 1), (10, 9), (32, 5)])
def test_thresholds_and_sizes(mq, K, L):
    from oracle import rates as R

    rng = np.random.default_rng(100 * K + L)
    U = np.asarray(W.cm(np.geomspace(20.0, 12000.0, K)))
    # thresholds u0 = E/2 of the pairs with level 0: a knot, just past it, below U_1, the last knot, above it
    special = [0.0, 2 * U[0], 2 * U[0] * (1 + 1e-13), 0.6 * U[0], 2 * U[-1], 2.4 * U[-1], 2 * U[K // 2]]
    E = np.array((special + list(rng.uniform(0.0, 1.9 * U[-1], 20)))[:L])
    g = 2.0 * rng.integers(0, 9, L) + 1.0
    # slowly varying positive values: every natural spline through them stays positive
    sig = 2.0 + np.sin(np.arange(K))[:, None, None] * rng.uniform(0.0, 0.2, (K, L, L)) + rng.uniform(0, 1, (1, L, L))
    kT = np.array([3.0, 30.0, 300.0, 3e4, 3e6]) * 3.1668115634556e-6
    sym, rate = mq.rate_coefficients(sig, U, E, g, 3000.0, kT)
    assert np.allclose(sym, R.sigma_sym(sig, g), rtol=1e-15, atol=0)
    ref = R.rates(sig, U, E, g, 3000.0, kT)
    ok = np.isfinite(ref) & (np.abs(ref) > 1e-250)
    assert ok.sum() > 0.2 * ok.size and np.all(np.isfinite(rate))
    assert np.max(np.abs(rate[ok] / ref[ok] - 1.0)) < 1e-10
    # excitations that the oracle underflows to zero (its quenching factor overflows to NaN instead)
    assert np.all(np.abs(rate[ref == 0.0]) < 1e-200)


def test_pairs_with_negative_or_nonfinite_values_take_the_quadrature(mq):
    """A tile that mixes pairs whose spline goes negative (clipped at zero), pairs with a NaN and ordinary
    pairs: the ordinary pairs keep their closed form, the others the clipped quadrature."""
    from oracle import rates as R

    K, L = 6, 12
    rng = np.random.default_rng(5)
    U = np.asarray(W.cm(np.geomspace(50.0, 5000.0, K)))
    E = np.sort(rng.uniform(0.0, float(U[-1]), L))
    g = np.ones(L)
    sig = np.full((K, L, L), 1.5) + rng.uniform(0.0, 0.1, (K, L, L))
    sig[:, 2, 3] = sig[:, 3, 2] = [1.0, 1.0, -1.0, -1.0, 1.0, 1.0]
    sig[3, 4, 5] = np.nan
    kT = np.array([300.0]) * 3.1668115634556e-6
    _, rate = mq.rate_coefficients(sig, U, E, g, 3000.0, kT)
    bad = np.zeros((L, L), bool)
    bad[4, 5] = bad[5, 4] = bad[2, 3] = bad[3, 2] = True
    ref = R.rates(np.where(np.isfinite(sig), sig, 1.0), U, E, g, 3000.0, kT)
    # a NaN knot makes every spline piece NaN, which the quadrature's max(v, 0) takes as zero
    assert 0.0 <= rate[0, 4, 5] < ref[0, 4, 5]
    # the panels do not resolve the kink where the spline crosses zero: about (panel width)^2
    assert abs(rate[0, 2, 3] / ref[0, 2, 3] - 1.0) < 1e-2
    assert np.max(np.abs(rate[0][~bad] / ref[0][~bad] - 1.0)) < 1e-10
