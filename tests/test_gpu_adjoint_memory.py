"""The adjoint short of device memory: down to the storage of counted steps, one state per step of a segment and one
thread block per SM it gives the same gradient; below, MQCT_ERR_OOM."""
import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu

ERR_OOM, SMS = 2, 152


def _gradient(mq, s, tr, dL, ckpt, limit):
    n = len(tr)
    w, g, out = np.ones(n), np.zeros(n, np.int32), np.zeros(s.n_params)
    st = mq.lib().mqct_probe_adjoint_limit(s.handle, tr.ctypes.data, n, w.ctypes.data, g.ctypes.data, 1, dL.ctypes.data, ckpt,
                                           out.ctypes.data, limit, None)
    return st, out


# the last one keeps its work vectors in global memory
@pytest.mark.parametrize("prec,jmax,n", [("fp64", 2, 400), ("fp32", 2, 400), ("fp32", 2, 3), ("fp32", 12, 330), ("fp64", 30, 20), ("fp32", 41, 310)])
@pytest.mark.parametrize("ckpt", [1, 16, 100000000])
def test_same_gradient_in_less_memory(prec, jmax, n, ckpt):
    import torch

    import paper_2312_02322_gb300.api as mq

    assert torch.cuda.get_device_properties(0).multi_processor_count == SMS
    s = mq.System.diatom(W.diatom_pes_params(jmax=jmax, n_grid=120), path="factorised", precision=prec, with_params=True)
    rng = np.random.default_rng(8)
    tr = np.zeros(n, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"] = W.cm(rng.uniform(2500.0, 3000.0, n)), rng.uniform(0.0, 2.0, n)
    tr["r0"], tr["r_end"], tr["dt"], tr["max_steps"] = (4.0, 4.0, 5.0, 100000) if jmax < 20 else (3.3, 3.3, 10.0, 100000)
    dL = rng.normal(size=(1, s.n_levels))
    _, _, d = mq.propagate(s, tr, want_pop=False, device=False)
    steps = int(d["steps"].max())
    assert np.all(d["status"] == 0) and steps > 10
    full = mq.adjoint(s, tr, np.ones(n), np.zeros(n, np.int32), 1, dL, ckpt=ckpt)
    # what the call takes at least: checkpoints and one segment of states for a block per SM
    size, amps = (8, 2) if prec == "fp64" else (4, 4)
    stride = (amps * s.n * size + 15) // 16 * 16 + 32
    K = min(ckpt, steps)
    vec = (17 * s.n + s.n_levels) * 2 * size
    vec_global = vec > 200000
    least = min(n, SMS) * ((steps // K + 2 + K) * stride + (((vec + 255) // 256 * 256) if vec_global else 0))
    for limit in (1 << 40, 8 * least, 4 * least, 3 * least // 2, least):
        st, g = _gradient(mq, s, tr, dL, ckpt, limit)
        assert st == 0
        assert np.max(np.abs(g - full)) <= 1e-12 * np.max(np.abs(full))
    assert _gradient(mq, s, tr, dL, ckpt, least - 1)[0] == ERR_OOM
