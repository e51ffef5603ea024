"""The adjoint refuses the trajectories that the propagation refuses, wherever in the call they stand, before any work
on the GPU."""
import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu

BAD = [("e_coll", np.inf), ("e_coll", 0.0), ("e_coll", 1e308), ("b", 6.0), ("b", -1.0), ("r0", 0.0),
       ("dt", 0.0), ("dt", np.nan), ("r_end", np.inf), ("max_steps", -1), ("init_state", -1), ("init_state", 9), ("system_idx", 1)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("field,value", BAD)
def test_refused_as_by_the_propagation(prec, field, value):
    import paper_2312_02322_gb300.api as mq

    s = mq.System.diatom(W.diatom_pes_params(jmax=2, n_grid=120), path="factorised", precision=prec, with_params=True)
    for where in (0, 2):
        tr = np.zeros(3, mq.TRAJ_DTYPE)
        tr["e_coll"], tr["b"], tr["r0"], tr["r_end"], tr["dt"], tr["max_steps"] = W.cm(2500.0), 1.0, 6.0, 6.0, 5.0, 10
        tr[field][where] = value
        with pytest.raises(mq.MQCTError) as fwd:
            mq.propagate(s, tr, device=False)
        with pytest.raises(mq.MQCTError) as adj:
            mq.adjoint(s, tr, np.ones(3), np.zeros(3, np.int32), 1, np.ones((1, s.n_levels)))
        assert fwd.value.status == adj.value.status == 1
