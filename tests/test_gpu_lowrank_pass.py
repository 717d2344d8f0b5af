"""The low-rank Hessian term's passes, H = diag(h0) + U diag(w) U^T without matrix rows: U^T v at
the numbers of columns where its block sums change their split, and its time for few columns.
"""
import numpy as np
import pytest

from paper_2405_03584_gb300 import ipm

pytestmark = pytest.mark.gpu


def _solver(n, cols):
    rng = np.random.default_rng(n + cols)
    U, w, h0 = rng.normal(size=(n, cols)) / np.sqrt(n), rng.uniform(0.1, 1.0, cols), rng.uniform(0.5, 2.0, n)
    s = ipm.Solver(precond="jacobi").set_qp(n, 0, rng.normal(size=n), None, np.zeros(n), np.full(n, np.inf), h0=h0, U=U, u_w=w)
    s.set_iterate(np.ones(n), np.zeros(0), np.zeros(0), np.full(n, 0.5), np.zeros(n), 0.1)
    return s, U, w, h0


# 1 .. 16 groups of 8 columns are added by 32 .. 2 threads a column, more by one
@pytest.mark.parametrize("n", [40, 20011])
@pytest.mark.parametrize("cols", [1, 2, 7, 8, 9, 16, 17, 24, 32, 33, 64, 65, 127, 128, 129, 136, 255, 256, 2049])
def test_columns(n, cols):
    if n * cols > 6_000_000:
        n = 3001
    s, U, w, h0 = _solver(n, cols)
    v = np.random.default_rng(5).normal(size=n)
    q = s.apply_kkt(v)                     # sigma = z_l / (x - l) = 0.5
    t = U.T @ v
    ref = (h0 + 0.5) * v + U @ (w * t)
    # every element is a sum of n products inside one of `cols`: their rounding, generously
    bound = 2.3e-16 * ((n + cols) * (np.abs(U) @ (w * (np.abs(U).T @ np.abs(v)))) + 8 * np.abs(ref))
    s.close()
    assert (np.abs(q - ref) <= bound).all()


@pytest.mark.parametrize("n,cols", [(1000, 1), (5000, 7), (20000, 7), (20000, 20)])
def test_few_columns_cost_no_more_than_many(n, cols):
    """The pass over few columns reads a fraction of what one over 64 reads."""
    def ms(c):
        s = _solver(n, c)[0]
        t = min(s.profile_operator(20)["ms_rows"] for _ in range(8))
        s.close()
        return t
    assert ms(cols) <= 1.2 * ms(64)
