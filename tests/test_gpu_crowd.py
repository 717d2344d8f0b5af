"""Many solves in one launch: what a solve's kernels cost beside others.

The solves of a batch share the float64 pipe, so a lane width that only pays while the chip is
otherwise idle must not make a batch slower than a narrower one.
"""
import time

import numpy as np
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


def test_one_member_more_takes_no_less():
    """A batch of 12 runs no slower form of the kernels than a batch of 13."""
    p = W.rt_qp(n=12000, density=0.005, seed=7)
    twelve = _batch_ms(p, 12, precond="jacobi_lr", storage="f32")
    assert twelve <= 1.01 * _batch_ms(p, 13, precond="jacobi_lr", storage="f32")


# the whole-chip form of the PCG's vector half: beyond 12 solves, above 4096 unknowns beyond 8, without
# the stiff rows' correction up to 2048 unknowns beyond 20
@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("precond,count,n", [("jacobi", 21, 200), ("jacobi", 13, 2100), ("jacobi", 9, 4400), ("jacobi_lr", 9, 4400)])
def test_same_bits_as_alone(precond, count, n, storage):
    solvers, ref = [], []
    for i in range(count):
        p = W.rt_qp(n=n + 37 * i, seed=60 + i, density=min(0.02, 12.0 / n))
        s = ipm.Solver(precond=precond, storage=storage, max_ipm=8)
        s.set_qp_rt(p)
        s.solve()
        ref.append(s.get())
        solvers.append(s)
    b = ipm.Batch(solvers)
    b.solve()
    for s, r in zip(solvers, ref):
        g = s.get()
        assert all(np.array_equal(g[k], r[k]) for k in ("x", "y", "zl", "zu", "s"))
        assert g["info"]["cg_iters"] == r["info"]["cg_iters"]
    b.close()
    for s in solvers:
        s.close()


def test_launch_counts():
    """A member's kernel_launches are those of the graph that ran: its own, or the batch's branch."""
    p = W.rt_qp(n=4400, density=0.003, seed=5)
    solvers = [ipm.Solver(precond="jacobi_lr") for _ in range(9)]
    for s in solvers:
        s.set_qp_rt(p)
    launches = lambda: [s.info()["kernel_launches"] for s in solvers]
    solvers[0].solve()
    alone = solvers[0].info()["kernel_launches"]
    b = ipm.Batch(solvers)
    b.solve()
    crowded = launches()
    assert len(set(crowded)) == 1 and crowded[0] > alone      # the whole-chip form has more launches
    for s in solvers:
        s.solve()
    assert launches() == [alone] * 9
    b.solve()
    assert launches() == crowded
    b.close()
    for s in solvers:
        s.close()
