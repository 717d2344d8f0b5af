"""The autotuner (options.autotune) where the column pass does not depend on the lane width.

H = diag(h0) + U diag(w) U^T without matrix rows and with an even number of columns runs its own
column kernel, so there is nothing to choose: the widths and the results are those of autotune = 0.
A choice made for another problem of the same size (an odd number of columns does use the
general column kernel) is not taken over.
"""
import numpy as np
import pytest

from paper_2405_03584_gb300 import ipm

pytestmark = pytest.mark.gpu


def _solver(n, cols, autotune):
    rng = np.random.default_rng(n)
    U = rng.normal(size=(n, cols)) / np.sqrt(n)
    s = ipm.Solver(autotune=autotune)
    return s.set_qp(n, 0, rng.normal(size=n), None, np.zeros(n), np.full(n, np.inf), h0=rng.uniform(0.5, 2.0, n), U=U,
                    u_w=rng.uniform(0.1, 1.0, cols))


@pytest.mark.parametrize("n", [500, 2000, 5001, 9001, 20000, 30011])
def test_low_rank_alone_keeps_its_width(n):
    ipm.autotune_reset()
    _solver(n, 7, 1).close()
    with _solver(n, 8, 0) as a, _solver(n, 8, 1) as b:
        assert b.get_config()["lanes_cols"] == a.get_config()["lanes_cols"]
        assert a.solve() == ipm.IPM_OK and b.solve() == ipm.IPM_OK
        assert np.array_equal(a.get()["x"], b.get()["x"])
    ipm.autotune_reset()
