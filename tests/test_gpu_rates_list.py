"""Rate coefficients of level sets that mix pairs in closed form with pairs that take the quadrature: each pair's rates are
those it has in a call of its own, whichever share of the pairs is listed, for more pairs than one pass takes, and
the listed pairs cost no more than if all were listed."""
import time

import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 2, 33, 150])
@pytest.mark.parametrize("nt", [1, 3, 64])
@pytest.mark.parametrize("share", [0.0, 0.01, 0.5, 1.0])
@pytest.mark.parametrize("sym", [True, False])
def test_pairs_alone_and_together(L, nt, share, sym):
    import paper_2312_02322_gb300.api as mq

    rng = np.random.default_rng(1000 * L + nt)
    K = 5
    U = np.asarray(W.cm(np.geomspace(50.0, 5000.0, K)))
    E = np.sort(rng.uniform(0.0, 2.2 * U[-1], L))  # some thresholds above the last energy
    g = 2.0 * rng.integers(0, 9, L) + 1.0
    sig = 1.0 + rng.uniform(0.0, 0.2, (K, L, L))
    sig[2] *= np.where(rng.random((L, L)) < share, -1.0, 1.0)
    kT = np.geomspace(20.0, 3000.0, nt) * 3.1668115634556e-6
    _, rate = mq.rate_coefficients(sig, U, E, g, 3000.0, kT, sigma_sym=sym)
    assert np.all(np.isfinite(rate)) and np.all(rate >= 0.0)
    for _ in range(12):
        a, b = np.sort(rng.integers(0, L, 2))
        i = [a, b] if a != b else [a]
        _, one = mq.rate_coefficients(sig[:, i][:, :, i], U, E[i], g[i], 3000.0, kT, sigma_sym=sym)
        assert np.array_equal(one, rate[:, i][:, :, i])


def test_more_pairs_than_one_pass():
    import torch

    import paper_2312_02322_gb300.api as mq

    L, K = 11700, 2
    gen = torch.Generator(device="cuda").manual_seed(3)
    sig = torch.rand((K, L, L), generator=gen, device="cuda", dtype=torch.float64)
    sig -= 0.05  # a tenth of the pairs is listed
    rng = np.random.default_rng(3)
    U, g = np.array([1e-3, 3e-3]), np.ones(L)
    E = np.sort(rng.uniform(0.0, 2e-3, L))
    kT = np.array([1e-3])
    _, rate = mq.rate_coefficients(sig, U, E, g, 3000.0, kT, sigma_sym=False)
    for rows in (np.arange(40), np.arange(L - 40, L), np.sort(rng.choice(L, 40, replace=False)), np.arange(11560, 11610)):
        i = torch.from_numpy(rows).cuda()
        sub = sig[:, i][:, :, i].cpu().numpy()
        _, one = mq.rate_coefficients(sub, U, E[rows], g[rows], 3000.0, kT, sigma_sym=False)
        assert np.array_equal(one, rate[:, i][:, :, i].cpu().numpy())


def test_listed_pairs_do_not_hold_the_others():
    import torch

    import paper_2312_02322_gb300.api as mq

    rs = W.rate_set(n_levels=200, temps_k=tuple(np.geomspace(10, 2000, 64)))
    rng = np.random.default_rng(0)
    sets = (rs.sigma * np.where(np.arange(10) % 3 == 1, -1.0, 1.0)[:, None, None],  # every pair
            np.where(rng.random(rs.sigma.shape) < 0.2, -0.3 * rs.sigma, rs.sigma))  # most pairs
    best = []
    for sig in sets:
        dev = torch.from_numpy(sig).cuda()
        times = []
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            mq.rate_coefficients(dev, rs.u, rs.energy, rs.g, rs.mu, rs.kT)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        best.append(min(times))
    assert best[1] < 1.2 * best[0]


def test_temperatures_cost_little_on_the_host():
    """A temperature adds its tables on the host and its kernel time to a call with five levels, far less than the
    microseconds that a temperature takes when every cosine of its series is evaluated anew."""
    import torch

    import paper_2312_02322_gb300.api as mq

    def best(nt):
        rs = W.rate_set(n_levels=5, temps_k=tuple(np.geomspace(10, 2000, nt)))
        dev = torch.from_numpy(rs.sigma).cuda()
        times = []
        for _ in range(30):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            mq.rate_coefficients(dev, rs.u, rs.energy, rs.g, rs.mu, rs.kT)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t0)
        return min(times)

    assert (best(256) - best(1)) / 255 < 3e-6
