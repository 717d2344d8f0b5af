"""Results copied to host memory: any subset of a call's vectors, at the sizes where the copies change
(16 KB for a single vector, 64 KB for one of several, 128 KB for an operand), equals what the device has; and a call moves
no more bytes than were asked for.
"""
import itertools
import json

import numpy as np
import pytest
import torch

from paper_2405_03584_gb300 import ipm, workloads as W

pytestmark = pytest.mark.gpu


def _call(name, s, want, device):
    """The requested outputs (dict name -> array) of one entry point."""
    n, m = s.n, s.m_rows
    sizes = {"get": dict(x=n, y=m, zl=n, zu=n, s=m), "resid": dict(rd=n, rp=m, rs=m, rl=n, ru=n),
             "dir": dict(dx=n, ds=m, dy=m, dzl=n, dzu=n)}[name]
    out = {k: (torch.full((c,), -7.0, dtype=torch.float64, device="cuda") if device else np.full(c, -7.0))
           for k, c in sizes.items() if k in want}
    ptr = lambda k: None if k not in out else (out[k].data_ptr() if device else out[k].ctypes.data)
    a = [ptr(k) for k in sizes]
    st, mem, L = ipm._default_stream(None), ipm.MEM_DEVICE if device else ipm.MEM_HOST, ipm.load()
    if name == "get":
        rc = L.ipm_get_xyz(s._h, *a, None, mem, st)
    elif name == "resid":
        kkt = np.full(4, -7.0)
        rc = L.ipm_residuals(s._h, *a, kkt.ctypes.data, mem, st)
        out["kkt"] = kkt
    else:
        rc = L.ipm_newton_direction(s._h, 1e-8, *a, None, mem, st)
    assert rc == ipm.IPM_OK
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() if torch.is_tensor(v) else v for k, v in out.items()}


def _solver(n, m):
    p = W.rt_qp(n=n, V=2 * max(n, m), density=min(1.0, 4.0 / n), n_organ=m, seed=n)
    s = ipm.Solver(precond="jacobi_lr", max_cg=20000)
    s.set_qp_rt(p)
    s.set_iterate(*W.random_iterate(n, m, p["l"], p["u"], 3, 1.0), 0.1)
    return s


@pytest.mark.parametrize("n,m", [(1, 1), (40, 90), (2047, 100), (2048, 2049), (2049, 30000), (8192, 50), (8193, 8192), (16384, 50), (16385, 16384), (30000, 17)])
def test_any_subset(n, m):
    s = _solver(n, m)
    for name, keys in (("get", "x y zl zu s"), ("resid", "rd rp rs rl ru"), ("dir", "dx ds dy dzl dzu")):
        keys = keys.split()
        ref = _call(name, s, keys, True)
        for r in (0, 1, 2, 4, 5):
            for want in itertools.combinations(keys, r):
                got = _call(name, s, want, False)
                assert all(np.array_equal(got[k], ref[k]) for k in want), (name, want)
                if name == "resid":
                    assert np.array_equal(got["kkt"], ref["kkt"])
    v = np.random.default_rng(n).normal(size=n)
    dv, dq = torch.from_numpy(v).cuda(), torch.empty(n, dtype=torch.float64, device="cuda")
    assert ipm.load().ipm_apply_kkt(s._h, dv.data_ptr(), dq.data_ptr(), ipm.MEM_DEVICE, ipm._default_stream(None)) == ipm.IPM_OK
    torch.cuda.synchronize()
    assert np.array_equal(s.apply_kkt(v), dq.cpu().numpy())
    s.close()


def _moved(f, tmp_path):
    """Bytes of the device-to-host copies of f."""
    f()
    for _ in range(2):                     # (a process's first profile records nothing)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            f()
            torch.cuda.synchronize()
    path = str(tmp_path / "trace.json")
    prof.export_chrome_trace(path)
    ev = [e for e in json.load(open(path))["traceEvents"] if e.get("cat") == "gpu_memcpy" and "DtoH" in e.get("name", "")]
    return sum(int(e["args"]["bytes"]) for e in ev)


def test_bytes_moved(tmp_path):
    n, m, scalars = 30000, 2000, 4096
    t = torch.zeros(1000, device="cuda")
    if _moved(lambda: t.cpu(), tmp_path) != 4000:
        pytest.skip("the profiler records no copies here")
    s = _solver(n, m)
    assert _moved(lambda: _call("get", s, ["x"], False), tmp_path) == 8 * n
    assert _moved(lambda: _call("get", s, [], False), tmp_path) == 0
    assert _moved(lambda: _call("get", s, ["y"], False), tmp_path) == 8 * m
    assert _moved(lambda: _call("resid", s, [], False), tmp_path) <= scalars
    assert _moved(lambda: _call("dir", s, ["dx"], False), tmp_path) <= 8 * n + scalars
    s.close()
    p = W.rt_two_sided(W.rt_qp(n=4000, density=0.003, seed=2))
    with ipm.Solver(precond="jacobi_lr", max_ipm=3) as s:
        s.set_qp_rt(p)
        s.solve()
        # x, z_l, z_u and the stored rows' y and s, once each, and what lies between them in the arena
        assert _moved(s.get, tmp_path) <= 8 * (3 * s.n + 2 * s.m_rows) + 2 * 16384
