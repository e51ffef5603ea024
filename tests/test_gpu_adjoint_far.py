"""A trajectory that is followed far beyond the distance it started from ends within the adjoint's checkpoint storage:
the call runs its kernel once."""
import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu


def _launches(mq, s, tr):
    g = mq.adjoint(s, tr, np.ones(len(tr)), np.zeros(len(tr), np.int32), 1, np.ones((1, s.n_levels)), ckpt=16)
    assert np.all(np.isfinite(g))
    return mq.last_launch_count()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("r0,r_end", [(6.0, 0.5), (6.0, 6.0), (6.0, 36.0), (3.5, 28.0), (4.0, 400.0)])
def test_one_run(prec, r0, r_end):
    import paper_2312_02322_gb300.api as mq

    s = mq.System.diatom(W.diatom_pes_params(jmax=2, n_grid=120), path="factorised", precision=prec, with_params=True)
    tr = np.zeros(3, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"], tr["r0"], tr["r_end"], tr["dt"] = W.cm(2500.0), [0.5, 1.0, 2.0], r0, r_end, 5.0
    tr["max_steps"] = 1000000
    far = _launches(mq, s, tr)
    tr["max_steps"] = 8  # never outruns its storage
    assert far == _launches(mq, s, tr)
