"""The FP64 kernel at the edges of its row groups and launch shapes: bases of 1 to 441 rows (fewer rows than a group
of 16, one more, several groups per warp), few trajectories and more than two per SM, both paths, a row whose
coupling is empty, against the oracle (the 1e-8 bar on probabilities; equal step counts and statuses)."""
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


@pytest.mark.parametrize("path", ["plain", "factorised"])
@pytest.mark.parametrize("jmax,n", [(0, 3), (1, 5), (3, 2), (3, 700), (4, 9), (6, 400), (9, 3), (15, 2), (20, 3)])
def test_sizes_and_shapes(mq, path, jmax, n):
    import oracle

    oracle.build()
    p = W.diatom_pes_params(jmax=jmax, n_grid=120)
    s = mq.System.diatom(p, path=path, precision="fp64")
    rng = np.random.default_rng(10 * jmax + n)
    tr = np.zeros(n, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"] = W.cm(rng.uniform(600.0, 2500.0, n)), rng.uniform(0.0, 4.0, n)
    tr["r0"], tr["r_end"], tr["dt"] = 7.0, 7.5, 5.0
    tr["max_steps"] = rng.integers(0, 61, n) if n > 100 else 5000
    tr["init_state"] = rng.integers(0, min(s.n, 9), n)
    pop, _, d = mq.propagate(s, tr, device=False)
    o = oracle.diatom_system(p.jmax, p.bconst, p.mu, p.A, p.beta, p.c6, p.rd, p.n_grid, p.r_min, p.r_max)
    for ms in np.unique(tr["max_steps"]):
        rows = np.flatnonzero(tr["max_steps"] == ms)
        amp, res = oracle.propagate(o, tr["e_coll"][rows], tr["b"][rows], tr["init_state"][rows], r0=7.0, r_end=7.5,
                                    dt=5.0, max_steps=int(ms))
        assert np.array_equal(d["steps"][rows], res["steps"])
        assert np.max(np.abs(pop[rows] - np.abs(amp) ** 2)) < 1e-8
    assert np.array_equal(d["status"] != 0, d["steps"] == tr["max_steps"])
    assert np.max(d["norm_dev"]) < 1e-6


@pytest.mark.parametrize("jmax,adapt,taken", [(47, None, True), (48, None, False), (41, (1e-8, 4), True), (42, (1e-8, 4), False)])
def test_largest_basis(mq, jmax, adapt, taken):
    """The FP64 path takes bases of up to 2387 rows or so (adaptive steps: 1790) and refuses larger ones."""
    p = W.diatom_pes_params(jmax=jmax, n_grid=60)
    s = mq.System.diatom(p, path="factorised", precision="fp64", adapt=adapt)
    tr = np.zeros(2, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"], tr["r0"], tr["r_end"], tr["dt"], tr["max_steps"] = W.cm(1000.0), 1.0, 7.0, 7.5, 5.0, 2
    if taken:
        _, _, d = mq.propagate(s, tr, device=False)
        assert np.all(d["steps"] > 0)
    else:
        with pytest.raises(mq.MQCTError):
            mq.propagate(s, tr, device=False)
