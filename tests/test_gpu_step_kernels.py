"""The kernels of the PCG iteration and of one interior point step at the sizes where their
splits change, against the oracle's formulas with the problem's matrices kept sparse.

* the iteration's vector half: one cluster of 8 or 16 blocks with 1, 2, 4 or 7 unknowns a
  thread (512 threads a block) up to 57344 unknowns (16384 without the stiff rows' correction),
  whole-chip kernels beyond;
* the low-rank correction by m stiff rows: chosen, ordered, their Gram matrix factored and
  inverted (a warp a column up to 256 rows, a block a column beyond), rows longer than 256
  entries;
* the low-rank Hessian term: even and odd column counts, more columns than a block covers at a
  time, alone (its own column kernel) and beside matrix rows;
* the triangular solves of the dense preconditioner, in blocks of 32 with the rows of a block
  two to a thread, even and odd sizes;
* the limit on PCG iterations with two iterations per pass of the loop;
* many solves in one launch.

A Newton direction is taken at eta = 1e-9: PCG stops at a residual of 1e-9 ||rhs|| by its own
recursion, and the true residual of the returned step may differ from the recursion's by what
the other tests allow an operator application (1e-10).  The rest of the direction follows from
dx by the oracle's recovery (every element a few float64 operations: 1e-10 of the largest).
"""
import types

import numpy as np
import pytest
import scipy.sparse as sp

from oracle import ipm as O
from paper_2405_03584_gb300 import ipm, workloads as W

pytestmark = pytest.mark.gpu

ETA, MU = 1e-9, 0.05


class LowRank:
    """diag(h0) + U diag(w) U^T."""

    def __init__(self, h0, U, w):
        self.h0, self.U, self.w = h0, U, w

    def __matmul__(self, v):
        return self.h0 * v + self.U @ (self.w * (self.U.T @ v))


def _qp(H, c, A, b, l, u):
    return types.SimpleNamespace(H=H, c=c, A=A, b=b, l=l, u=u, n=len(c), m=A.shape[0], fl=np.isfinite(l), fu=np.isfinite(u))


def _rt(n, V=None, per_row=6.0, m=None, seed=1):
    p = W.rt_qp(n=n, V=V, density=min(1.0, per_row / n), n_organ=m, seed=seed)
    D = sp.csr_matrix((p["D_data"], p["D_indices"], p["D_indptr"]), shape=(p["V"], n))
    H = (D.T @ sp.diags(p["w"]) @ D + sp.diags(p["h0"])).tocsr()
    return p, _qp(H, p["c"], D[p["a_rows"]], p["b"], p["l"], p["u"])


def _low_rank(n, cols, rows, seed):
    rng = np.random.default_rng(seed)
    U = rng.normal(size=(n, cols)) / np.sqrt(n)
    w = rng.uniform(0.1, 1.0, size=cols)
    h0 = rng.uniform(0.5, 2.0, size=n)
    A = sp.random(rows, n, density=min(1.0, 5.0 / n), random_state=seed, format="csr") if rows else sp.csr_matrix((0, n))
    qp = _qp(LowRank(h0, U, w), rng.normal(size=n), A, np.ones(rows), np.zeros(n), np.full(n, np.inf))
    s = lambda **o: ipm.Solver(**o).set_qp(n, rows, qp.c, qp.b, qp.l, qp.u, h0=h0, U=U, u_w=w, A=(
        A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data) if rows else None)
    return qp, s


def _check(s, qp, eta=ETA, tol=ETA + 1e-10):
    x, sl, y, zl, zu = W.random_iterate(qp.n, qp.m, qp.l, qp.u, 7, 1.0)
    it = O.Iterate(x, sl, y, zl, zu)
    res = O.residuals(qp, it, MU)
    rd, rp, rs, rl, ru = res
    tl, tu = O._tl(qp, x), O._tu(qp, x)
    theta = y / sl
    sigma = np.where(qp.fl, zl / tl, 0.0) + np.where(qp.fu, zu / tu, 0.0)
    K = lambda v: qp.H @ v + qp.A.T @ (theta * (qp.A @ v)) + sigma * v
    rhs = -rd - np.where(qp.fl, rl / tl, 0.0) + np.where(qp.fu, ru / tu, 0.0) - qp.A.T @ (theta * rp - rs / sl)
    s.set_iterate(x, sl, y, zl, zu, MU)
    g = s.residuals()
    close = lambda a, b: np.testing.assert_allclose(a, b, rtol=1e-10, atol=1e-10 * (np.abs(b).max() if b.size else 1.0))
    close(g["rd"], rd)
    close(g["rp"], rp)
    v = np.random.default_rng(5).normal(size=qp.n)
    close(s.apply_kkt(v), K(v))
    d = s.newton_direction(eta=eta)
    assert d["report"]["converged"] == 1, d["report"]
    assert np.linalg.norm(K(d["dx"]) - rhs) <= tol * np.linalg.norm(rhs)
    ref = O.recover_direction(qp, it, res, d["dx"])
    for k, r in (("ds", ref.s), ("dy", ref.y), ("dzl", ref.zl), ("dzu", ref.zu)):
        close(d[k], r)
    return d["report"]


# 512 (last system of 8 blocks), 8192, 16384, 32768, 57344 (last of 1, 2, 4, 7 unknowns a thread)
@pytest.mark.parametrize("precond", ["jacobi", "jacobi_lr"])
@pytest.mark.parametrize("n", [1, 33, 512, 513, 8192, 8193, 16385, 32769, 57344, 57345])
def test_vector_half_sizes(n, precond):
    p, qp = _rt(n, V=2 * n, m=max(1, n // 10))
    with ipm.Solver(precond=precond, max_cg=20000) as s:
        s.set_qp_rt(p)
        _check(s, qp)


@pytest.mark.parametrize("m,per_row", [(1, 6.0), (31, 6.0), (33, 300.0), (64, 6.0), (65, 6.0), (129, 6.0), (256, 6.0),
                                       (257, 6.0), (400, 300.0)])
def test_stiff_rows(m, per_row):
    p, qp = _rt(1501, V=1300, per_row=per_row, m=m, seed=m)
    with ipm.Solver(precond="jacobi_lr", max_cg=20000, stiff_max=512, stiff_gamma=1e-12) as s:
        s.set_qp_rt(p)
        assert _check(s, qp)["stiff_rows"] == m


@pytest.mark.parametrize("n,cols,rows", [(1, 2, 0), (64, 1, 0), (65, 34, 0), (1000, 7, 0), (1000, 200, 0), (130, 2050, 0),
                                         (130, 2051, 0), (57345, 6, 0), (65, 34, 40), (1000, 7, 300), (57345, 6, 100)])
def test_low_rank_hessian(n, cols, rows):
    qp, make = _low_rank(n, cols, rows, seed=n + cols)
    with make(precond="jacobi", max_cg=20000) as s:
        _check(s, qp)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 545, 577])
def test_dense_solves(n):
    p = W.dense_qp(n=n, m=2 * n, seed=n)
    qp = O.from_dense(p)
    with ipm.Solver(precond="dense") as s:
        s.set_qp_dense(p["H"], p["c"], p["A"], p["b"], p["l"], p["u"])
        assert _check(s, qp)["iters"] <= 4


@pytest.mark.parametrize("limit", [1, 2, 3])
def test_iteration_limit(limit):
    p, qp = _rt(1501)
    x, sl, y, zl, zu = W.random_iterate(qp.n, qp.m, qp.l, qp.u, 7, 1.0)
    with ipm.Solver(precond="jacobi", max_cg=limit) as s:
        s.set_qp_rt(p)
        s.set_iterate(x, sl, y, zl, zu, MU)
        rep = s.newton_direction(eta=1e-14)["report"]
    assert rep["iters"] == limit and rep["converged"] == 0


# more than 12 solves in one launch take the whole-chip form of the vector half
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_many_solves_in_one_launch(storage):
    """13 uneven QPs in one launch give each member the bits of its solve alone."""
    solvers, ref = [], []
    for i in range(13):
        p = W.rt_qp(n=200 + 37 * i, seed=60 + i, density=0.02, n_organ=60 + 5 * i)
        s = ipm.Solver(precond="jacobi_lr", storage=storage)
        s.set_qp_rt(p)
        assert s.solve() == ipm.IPM_OK
        ref.append(s.get()["x"])
        solvers.append(s)
    b = ipm.Batch(solvers)
    assert b.solve() == [ipm.IPM_OK] * 13
    for s, x in zip(solvers, ref):
        assert np.array_equal(s.get()["x"], x)
    b.close()
    for s in solvers:
        s.close()
