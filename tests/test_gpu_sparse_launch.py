"""The sparse stage kernel on either side of its launch rule (a grid that four thread blocks per SM hold, or a larger
one): the same bits for the same trajectories."""
import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 100, 2048, 2784])  # N = 1681: seven row blocks, so 7, 28, 448 and 609 thread blocks
def test_both_forms_agree(n):
    import paper_2312_02322_gb300.api as mq

    trunc = (float(W.cm(W.PAPER_TRUNC_CM)), *W.PAPER_TRUNC_R)
    s = mq.System.diatom(W.sparse_pes_params(jmax=40, lam_max=6), path="plain", precision="fp32", grid="log", trunc=trunc)
    rng = np.random.default_rng(3)
    tr = np.zeros(4096, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"] = W.cm(rng.uniform(600.0, 3000.0, 4096)), rng.uniform(0.0, 5.0, 4096)
    tr["r0"], tr["r_end"], tr["dt"], tr["max_steps"] = 9.0, 60.0, 5.0, 20
    ref, _, d = mq.propagate(s, tr, device=False)  # 896 thread blocks
    pop, _, e = mq.propagate(s, tr[:n].copy(), device=False)
    assert np.all(np.isfinite(ref)) and np.array_equal(pop, ref[:n]) and np.array_equal(e["steps"], d["steps"][:n])
