"""A bounded device wait that runs out (made to run out when a thread block claims every `fail_every`-th item of the
work list): the trajectories the block then holds get MQCT_TRAJ_TIMEOUT and NaN results, all others the results of
an ordinary call, and the call and the next one end."""
import ctypes as C

import numpy as np
import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu

ERR_TIMEOUT, TIMEOUT = 5, 8


def _call(systems, tr, fail_every, shape=0, device=False, diag=True):
    """mqct_probe_propagate_timeout: (status, pop, amp, diag)"""
    import torch

    import paper_2312_02322_gb300.api as mq

    systems = systems if isinstance(systems, list) else [systems]
    n, nmax = len(tr), max(s.n for s in systems)
    hs = (C.c_void_p * len(systems))(*[s.handle.value for s in systems])
    op = mq.PropagateOpts()
    shapes = np.full(len(systems), shape, np.int32)
    op.batch_shape = shapes.ctypes.data
    pop, amp, d = np.zeros((n, nmax)), np.zeros((n, nmax, 2)), np.zeros(n, mq.DIAG_DTYPE)
    if device:
        tp = torch.zeros((n, nmax), dtype=torch.float64, device="cuda")
        dt = torch.from_numpy(tr.view(np.uint8).copy()).cuda()
        st = mq.lib().mqct_probe_propagate_timeout(hs, len(systems), dt.data_ptr(), n, tp.data_ptr(), None, None, C.byref(op),
                                                   fail_every, torch.cuda.current_stream().cuda_stream)
        return st, tp.cpu().numpy(), None, None
    st = mq.lib().mqct_probe_propagate_timeout(hs, len(systems), tr.ctypes.data, n, pop.ctypes.data, amp.ctypes.data,
                                               d.ctypes.data if diag else None, C.byref(op), fail_every, None)
    return st, pop, amp, d


def _trajs(mq, n, cap, seed):
    rng = np.random.default_rng(seed)
    tr = np.zeros(n, mq.TRAJ_DTYPE)
    tr["e_coll"], tr["b"] = W.cm(rng.uniform(600.0, 2500.0, n)), rng.uniform(0.0, 4.0, n)
    tr["r0"], tr["r_end"], tr["dt"], tr["max_steps"] = 7.0, 50.0, 5.0, rng.integers(0, cap + 1, n)
    return tr


def _check(mq, systems, tr, fail_every, **kw):
    """the trajectories that timed out"""
    st, pop, amp, d = _call(systems, tr, fail_every, **kw)
    ref, ramp, e = mq.propagate(systems, tr, want_amp=True, device=False, batch_shape=kw.get("shape", 0))
    out = (d["status"] & TIMEOUT) != 0
    nst = np.array([s.n for s in (systems if isinstance(systems, list) else [systems])])[tr["system_idx"]]
    used = np.arange(pop.shape[1])[None, :] < nst[:, None]
    assert st == (ERR_TIMEOUT if out.any() else 6)
    assert np.all(np.isnan(pop[out][used[out]])) and np.all(np.isnan(amp[out][used[out]]))
    assert np.array_equal(d["steps"][~out], e["steps"][~out]) and np.array_equal(d["status"][~out], e["status"][~out])
    ok = used & ~out[:, None]
    assert np.max(np.abs(np.where(ok, pop - ref, 0.0))) < 1e-6
    assert np.max(np.abs(np.where(ok, amp[..., 0] + 1j * amp[..., 1] - ramp, 0.0))) < 1e-6
    return out


@pytest.mark.parametrize("shape", [0, 1, 3, 5, 7])
@pytest.mark.parametrize("fail_every", [0, 1, 77, 1500, 4000])
def test_fp32_block_goes_on(shape, fail_every):
    import paper_2312_02322_gb300.api as mq

    s = mq.System.diatom(W.diatom_pes_params(jmax=6, n_grid=120), path="factorised", precision="fp32")
    tr = _trajs(mq, 6000, 20, 3)
    out = _check(mq, s, tr, fail_every, shape=shape)
    # every claim ends its block's trajectories, or the blocks that make the others claim go on
    assert out.all() if fail_every == 1 else (out.any() == (fail_every > 0) and not out.all())
    few = tr[:7].copy()
    assert _check(mq, s, few, 1, shape=shape).all() and not _check(mq, s, few, 8, shape=shape).any()


def test_fp32_several_systems():
    import paper_2312_02322_gb300.api as mq

    ss = [mq.System.diatom(W.diatom_pes_params(jmax=j, n_grid=120), path="factorised", precision="fp32") for j in (2, 20, 9)]
    tr = _trajs(mq, 4000, 20, 4)
    tr["system_idx"] = np.random.default_rng(5).integers(0, 3, len(tr))
    for fail_every in (1, 5, 400):
        out = _check(mq, ss, tr, fail_every)
        assert out.all() if fail_every == 1 else 0 < out.sum() < len(tr)


def test_fp32_without_diagnostics():
    """Device outputs and no diagnostics: the NaN rows tell."""
    import paper_2312_02322_gb300.api as mq

    s = mq.System.diatom(W.diatom_pes_params(jmax=3, n_grid=120), path="factorised", precision="fp32")
    tr = _trajs(mq, 9, 20, 6)
    st, pop, _, _ = _call(s, tr, 1, device=True)
    assert st == 0 and np.all(np.isnan(pop))
    st, pop, _, _ = _call(s, tr, 0, device=True)
    assert st == 0 and np.all(np.isfinite(pop))
    # host outputs and no diagnostics: the status of the call
    assert _call(s, tr, 1, diag=False)[0] == ERR_TIMEOUT


@pytest.mark.parametrize("path", ["plain", "factorised"])
@pytest.mark.parametrize("adapt", [None, (1e-6, 4)])
@pytest.mark.parametrize("jmax,n", [(2, 1000), (13, 200)])
def test_fp64_trajectory_alone_is_void(path, adapt, jmax, n):
    import paper_2312_02322_gb300.api as mq

    s = mq.System.diatom(W.diatom_pes_params(jmax=jmax, n_grid=120), path=path, precision="fp64", adapt=adapt)
    tr = _trajs(mq, n, 20, 7)
    for fail_every in (0, 1, 3, n, n + 1):
        assert _check(mq, s, tr, fail_every).sum() == (n // fail_every if fail_every else 0)


def test_fp64_without_diagnostics():
    import paper_2312_02322_gb300.api as mq

    s = mq.System.diatom(W.diatom_pes_params(jmax=3, n_grid=120), path="plain", precision="fp64")
    tr = _trajs(mq, 9, 20, 6)
    st, pop, _, _ = _call(s, tr, 2, device=True)
    assert st == 0 and np.all(np.isnan(pop), axis=1).sum() == 4 and np.isnan(pop).sum() == 4 * s.n
    assert _call(s, tr, 2, diag=False)[0] == ERR_TIMEOUT
