"""Lanes per row and per column of the float64 operator passes (no width asked for, no autotuner).

Each shape with the widths that were measured fastest on it, or within a few percent of that:
long rows in a matrix too small to fill the chip (a dense block), short columns in a wide matrix,
and the shapes of the RT and dense workloads.
"""
import numpy as np
import pytest

from paper_2405_03584_gb300 import ipm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n,per_row,lanes_rows,lanes_cols", [
    (4096, 2048, 2048, 32, 32), (8192, 4096, 512, 16, 32), (8192, 4096, 1024, 16, 32), (2048, 1024, 1024, 32, 32),
    (1000, 50000, 2500, 32, 4), (500, 20000, 4000, 32, 8), (40000, 10000, 100, 4, 16),
    (28004, 7001, 42, 4, 16), (48000, 12000, 60, 4, 8), (80000, 20000, 60, 4, 16), (36000, 9000, 20, 4, 8), (4400, 1100, 4, 4, 8), (6000, 1500, 9, 4, 16), (1000, 500, 500, 32, 32), (16000, 1000, 500, 8, 32)])
def test_widths(rows, n, per_row, lanes_rows, lanes_cols):
    rng = np.random.default_rng(1)
    first = rng.integers(0, n - per_row + 1, rows)
    idx = (first[:, None] + np.arange(per_row)).astype(np.int32).ravel()
    F = (np.arange(rows + 1, dtype=np.int64) * per_row, idx, rng.uniform(0.5, 1.5, rows * per_row))
    with ipm.Solver(precond="jacobi") as s:
        s.set_qp(n, 0, np.zeros(n), None, np.zeros(n), np.ones(n), h0=np.ones(n), F=F, f_w=np.ones(rows))
        cfg = s.get_config()
    assert (cfg["lanes_rows"], cfg["lanes_cols"]) == (lanes_rows, lanes_cols)
