"""The PCG's vector half with the reduced storages, and with the stiff rows' correction in use, at the
sizes where its form changes: 1, 2, 4 or 7 unknowns a thread of the cluster kernel (up to 8192,
16384, 32768 and 57344 unknowns), the whole-chip kernels beyond.

A direction of a reduced storage is held to the same residual as a float64 one: both refinement
schemes end on the float64 residual (1e-9 of the right-hand side, plus the 1e-10 that the float64
operator is allowed elsewhere).
"""
import pytest

from tests.test_gpu_step_kernels import _check, _rt
from paper_2405_03584_gb300 import ipm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [512, 513, 8192, 8193, 16385, 32769, 57344, 57345])
def test_stiff_rows_in_use(n):
    p, qp = _rt(n, V=2 * n, m=max(60, n // 10))
    with ipm.Solver(precond="jacobi_lr", max_cg=20000) as s:
        s.set_qp_rt(p)
        assert _check(s, qp)["stiff_rows"] > 0


@pytest.mark.parametrize("refine_mode", [0, 1])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("precond", ["jacobi", "jacobi_lr"])
@pytest.mark.parametrize("n", [4097, 8193, 16385, 32769, 57345])
def test_reduced_storage(n, precond, storage, refine_mode):
    p, qp = _rt(n, V=2 * n, m=n // 10)
    with ipm.Solver(precond=precond, storage=storage, refine_mode=refine_mode, refine_max=30, max_cg=20000) as s:
        s.set_qp_rt(p)
        rep = _check(s, qp)
        assert precond == "jacobi" or rep["stiff_rows"] > 0


# more stiff rows than the 256 warps of a cluster: a warp takes a second row, and fetches the first again
@pytest.mark.parametrize("refine_mode", [0, 1])
@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("m,per_row", [(257, 6.0), (400, 300.0)])
def test_many_stiff_rows(m, per_row, storage, refine_mode):
    p, qp = _rt(1501, V=1300, per_row=per_row, m=m, seed=m)
    with ipm.Solver(precond="jacobi_lr", storage=storage, refine_mode=refine_mode, refine_max=30, max_cg=20000, stiff_max=512,
                    stiff_gamma=1e-12) as s:
        s.set_qp_rt(p)
        assert _check(s, qp)["stiff_rows"] == m
