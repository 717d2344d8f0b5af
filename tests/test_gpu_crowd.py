"""Many solves in one launch: what a solve's kernels cost beside others.

The solves of a batch share the float64 pipe, so a lane width that only pays while the chip is
otherwise idle must not make a batch slower than a narrower one.
"""
import time

import pytest

from paper_2405_03584_gb300 import ipm, workloads as W

pytestmark = pytest.mark.gpu


def _batch_ms(p, count, **opts):
    first = ipm.Solver(**opts)
    first.set_qp_rt(p)
    solvers = [first] + [ipm.Solver(**opts).share_qp(first) for _ in range(count - 1)]
    b = ipm.Batch(solvers)
    best = 1e30
    for _ in range(5):
        t0 = time.perf_counter()
        assert b.solve() == [ipm.IPM_OK] * count
        best = min(best, time.perf_counter() - t0)
    b.close()
    for s in reversed(solvers):
        s.close()
    return 1e3 * best


def test_default_width_in_a_batch():
    p = W.rt_qp(n=12000, density=0.005, seed=7)
    narrow = _batch_ms(p, 16, precond="jacobi_lr", lanes_cols=8)
    assert _batch_ms(p, 16, precond="jacobi_lr") <= 1.06 * narrow
