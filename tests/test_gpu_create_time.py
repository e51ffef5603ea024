"""Creating a system for the FP32 batched kernel takes little longer than creating the FP64 one: its group tables cost a
pass over the coupling, and a basis that no launch shape takes has none."""
import time

import pytest

import paper_2312_02322_gb300.inputs as W

pytestmark = pytest.mark.gpu


def _best(make, reps):
    times = []
    for _ in range(reps):
        t0 = time.perf_counter()
        make().close()
        times.append(time.perf_counter() - t0)
    return min(times)


def test_fp32_tables_cost_little():
    import paper_2312_02322_gb300.api as mq

    p = W.asym_pes_params(jmax=8)  # 28 terms
    fp64, fp32 = (_best(lambda: mq.System.asym_top(p, path="factorised", precision=q), 7) for q in ("fp64", "fp32"))
    assert fp32 < 1.07 * fp64  # 1.10 when every two terms were compared row by row
    q = W.diatom_pes_params(jmax=60, n_grid=400)  # 3721 rows
    fp64, fp32 = (_best(lambda: mq.System.diatom(q, path="factorised", precision=x), 9) for x in ("fp64", "fp32"))
    assert fp32 < 1.1 * fp64
