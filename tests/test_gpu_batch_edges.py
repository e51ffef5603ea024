"""The FP32 batched kernel at the edges of its tiles: bases of one row to the largest that fits, around the
rows a CTA's element threads cover, one to six expansion terms (identity only, an unpaired group, pairs), every
launch shape, step counts from 0 upwards with more trajectories than slots, against the FP64 kernel (the 1e-4
bar on probabilities of the mixed path; equal step counts, which max_steps sets here)."""
import dataclasses

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


def _params(jmax, terms):
    p = W.diatom_pes_params(jmax=jmax, n_grid=120)
    A = np.concatenate([p.A, [W.cm(1.5e3)]])[:terms]
    beta = np.concatenate([p.beta, [2.3]])[:terms]
    return dataclasses.replace(p, A=A, beta=beta)


def _trajs(mq, sys_, n, cap, seed):
    rng = np.random.default_rng(seed)
    tr = np.zeros(n, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"] = W.cm(rng.uniform(600.0, 2500.0, n)), rng.uniform(0.0, 4.0, n)
    tr["r0"], tr["r_end"], tr["dt"] = 7.0, 50.0, rng.choice([4.0, 5.0], n)
    tr["max_steps"] = rng.integers(0, cap + 1, n)
    tr["init_state"] = rng.integers(0, min(sys_.n, 9), n)
    return tr


def _compare(mq, params, tr, systems_of, **opt):
    pop, amp, d = mq.propagate(systems_of("fp32"), tr, want_amp=True, device=False, **opt)
    ref, ramp, e = mq.propagate(systems_of("fp64"), tr, want_amp=True, device=False)
    assert np.array_equal(d["steps"], e["steps"]) and np.array_equal(d["status"], e["status"])
    assert np.max(np.abs(pop - ref)) < 1e-4 and np.max(np.abs(amp - ramp)) < 1e-4
    assert np.max(d["norm_dev"]) < 1e-5 and np.max(d["energy_dev"] / tr["e_coll"]) < 1e-4


@pytest.mark.parametrize("jmax,terms,shape", [
    (0, 1, 0), (0, 5, 1), (1, 2, 2), (4, 3, 3), (5, 6, 4),      # 1, 4, 25, 36 rows
    (13, 5, 7), (14, 5, 7), (14, 4, 3),                         # 196, 225: one and two units per thread
    (20, 5, 4), (20, 5, 7), (21, 5, 4), (21, 6, 5),             # 441, 484: past the widest slot count
    (29, 2, 5), (42, 5, 0), (41, 1, 2),                         # 900, 1849, 1764
])
def test_sizes_terms_and_shapes(mq, jmax, terms, shape):
    p = _params(jmax, terms)
    sys_ = {q: mq.System.diatom(p, path="factorised", precision=q) for q in ("fp32", "fp64")}
    n, cap = (41, 120) if jmax < 30 else (13, 40)
    _compare(mq, p, _trajs(mq, sys_["fp64"], n, cap, 7 * jmax + terms), sys_.get, batch_shape=shape)


def test_more_trajectories_than_slots(mq):
    """Every slot of the GPU is refilled at least once, at different times."""
    p = _params(6, 5)
    sys_ = {q: mq.System.diatom(p, path="factorised", precision=q) for q in ("fp32", "fp64")}
    _compare(mq, p, _trajs(mq, sys_["fp64"], 3000, 60, 3), sys_.get, batch_shape=7)


def test_systems_of_one_call(mq):
    """CTAs that bind to one system after the other, with other slot counts and groups."""
    ps = [_params(j, t) for j, t in ((2, 5), (20, 1), (9, 4), (30, 5))]
    sys_ = {q: [mq.System.diatom(p, path="factorised", precision=q) for p in ps] for q in ("fp32", "fp64")}
    rng = np.random.default_rng(5)
    tr = np.concatenate([_trajs(mq, sys_["fp64"][s], 60, 50, 11 + s) for s in range(4)])
    tr["system_idx"] = np.repeat(np.arange(4), 60)
    tr = tr[rng.permutation(len(tr))].copy()
    nst = np.array([s.n for s in sys_["fp64"]])[tr["system_idx"]]
    for shape in (0, 2, 5):
        pop, _, d = mq.propagate(sys_["fp32"], tr, device=False, batch_shape=shape)
        ref, _, e = mq.propagate(sys_["fp64"], tr, device=False)
        used = np.arange(pop.shape[1])[None, :] < nst[:, None]
        assert np.array_equal(d["steps"], e["steps"]) and np.array_equal(d["status"], e["status"])
        assert np.max(np.abs(np.where(used, pop - ref, 0.0))) < 1e-4
