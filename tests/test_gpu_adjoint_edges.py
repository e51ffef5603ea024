"""The adjoint's stored stage states: with a checkpoint interval whose segments would outgrow their storage the stage states are
recomputed instead; both give the same gradient to rounding (the same arithmetic)."""
import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("jmax", [1, 4])
def test_recomputed_and_stored_stages_agree(prec, jmax):
    import paper_2312_02322_gb300.api as mq

    p = W.diatom_pes_params(jmax=jmax, n_grid=120)
    s = mq.System.diatom(p, path="factorised", precision=prec, with_params=True)
    tr = np.zeros(1, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"], tr["r0"], tr["r_end"], tr["dt"], tr["max_steps"] = W.cm(2500.0), 1.0, 6.0, 6.0, 5.0, 100000
    dL = np.random.default_rng(3).normal(size=(1, s.n_levels))
    args = (s, tr, np.ones(1), np.zeros(1, np.int32), 1, dL)
    stored = mq.adjoint(*args, ckpt=16)
    # a step and its stage states take at least 40 n bytes: segments of more than 16 GB with them
    recomputed = mq.adjoint(*args, ckpt=(18 << 30) // (40 * s.n))
    assert np.linalg.norm(stored) > 0
    assert np.max(np.abs(stored - recomputed)) <= 1e-12 * np.max(np.abs(stored))


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_trajectory_that_outruns_its_checkpoints(prec):
    """r_end far beyond r0: more steps than three free flights of 2 r0, so the call counts them and runs again; the
    same gradient as with an interval that needs no second checkpoint."""
    import paper_2312_02322_gb300.api as mq

    p = W.diatom_pes_params(jmax=2, n_grid=120)
    s = mq.System.diatom(p, path="factorised", precision=prec, with_params=True)
    tr = np.zeros(3, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"], tr["r0"], tr["r_end"] = W.cm(2500.0), [0.5, 1.0, 2.0], 6.0, [6.0, 60.0, 6.0]
    tr["dt"], tr["max_steps"] = 5.0, 100000
    dL = np.random.default_rng(4).normal(size=(1, s.n_levels))
    args = (s, tr, np.ones(3), np.zeros(3, np.int32), 1, dL)
    many, one = mq.adjoint(*args, ckpt=16), mq.adjoint(*args, ckpt=20000)
    assert np.linalg.norm(one) > 0
    assert np.max(np.abs(many - one)) <= 1e-12 * np.max(np.abs(one))
