"""Rows that repeat a column: the operator adds the entries up, and so does the stiff rows' correction.

(The interface asks for rows without repeats; such rows are not checked for and solve as the summed
entries' do, if in more iterations: the Jacobi diagonal takes each entry's square.)
"""
import numpy as np
import pytest

from paper_2405_03584_gb300 import ipm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,density", [(600, 0.03), (1500, 0.01), (4000, 0.01)])
def test_solves(n, density):
    p = W.rt_qp(n=n, density=density, seed=21)
    q = dict(p)
    part = np.random.default_rng(0).uniform(0.1, 0.9, len(p["D_data"]))
    q.update(D_indptr=2 * p["D_indptr"], D_indices=np.repeat(p["D_indices"], 2),
             D_data=np.stack([part * p["D_data"], (1 - part) * p["D_data"]], 1).ravel())
    obj = []
    for z in (p, q):
        with ipm.Solver(precond="jacobi_lr") as s:
            s.set_qp_rt(z)
            assert s.solve() == ipm.IPM_OK
            i = s.info()
            assert i["max_stiff_rows"] > 0
            obj.append(i["primal_obj"])
    assert abs(obj[0] - obj[1]) <= 2e-6 * (1 + abs(obj[0]))      # both within rel. KKT 1e-6 of the optimum
