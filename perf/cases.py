"""Timed cases of the interior point library, over the range of sizes it is used at.

A case is one call (or one short sequence of calls) of ``paper_2405_03584_gb300.ipm`` on a QP
of one of the shapes this repository generates in ``workloads``:

* ``rt``    radiation-therapy QP: H = D^T diag(w) D + 1e-4 I with D voxels x spots (4 n rows of
            a few contiguous bands), constraint rows = rows of D, 0 <= x <= 5;
* ``dense`` dense QP: H = Q diag(lam) Q^T, dense A, 0 <= x <= 10;
* ``bfgs``  quasi-Newton sub-problem: H = diag(h0) + U W U^T with 2 k columns, x >= 0, and
            optionally banded constraint rows (the proton shape has none, the VMAT shape has).

The calls (``op``):

* ``solve``  a whole cold solve and the copy of its result to the host;
* ``serve``  new costs for the loaded plan, then as ``solve`` (a served request);
* ``batch``  several QPs of uneven sizes in one launch, and their results;
* ``dir``    one Newton direction (residuals, preconditioner, right-hand side, PCG, recovery);
* ``apply``  one application of the PCG operator;
* ``resid``  the KKT residuals of the current point.

The single-step calls run at a random strictly interior point.  Inputs are drawn on the GPU;
sums that enter them are integer sums, so a seed gives the same bits in every process.
"""
import math

import numpy as np
import torch

from paper_2405_03584_gb300 import ipm


def listed():
    return [
        # the smallest Newton step: every launch and every gap between launches counts
        dict(name="dir_dense_24", kind="dense", op="dir", n=24, m=48, eta=1e-12),
        # the dense workload of the benchmark (C0): a step with its factorisation
        dict(name="dir_dense_500", kind="dense", op="dir", n=500, m=1000, eta=1e-12),
        # a small plan with few entries a row
        dict(name="solve_rt_1500", kind="rt", op="solve", n=1500, nnz_row=9.0, organ=0.1, storage="f64"),
        # a request on a plan of the serving mix: odd size, half as many constraint rows as variables
        dict(name="serve_rt_7001", kind="rt", op="serve", n=7001, nnz_row=42.0, organ=0.125, storage="f64"),
        # uneven QPs in one launch, in the batch's storage
        dict(name="batch_rt_8", kind="rt", op="batch", n=12000, count=8, nnz_row=60.0, organ=0.125, storage="f32"),
        # one of its larger members alone
        dict(name="solve_rt_12007_f32", kind="rt", op="solve", n=12007, nnz_row=48.0, organ=0.125, storage="f32"),
        # one accurate Newton step at a given point
        dict(name="dir_rt_10007", kind="rt", op="dir", n=10007, nnz_row=50.0, organ=0.1, storage="f64", eta=1e-13),
        # the full-size plan: one application of the operator, the whole solve in both storages in use
        dict(name="apply_rt_50000", kind="rt", op="apply", n=50000, nnz_row=250.0, organ=0.1, storage="f64"),
        dict(name="solve_rt_50000", kind="rt", op="solve", n=50000, nnz_row=250.0, organ=0.1, storage="f64"),
        dict(name="solve_rt_50000_bf16", kind="rt", op="solve", n=50000, nnz_row=250.0, organ=0.1, storage="bf16"),
        # quasi-Newton sub-problems in the proton and the VMAT shape
        dict(name="solve_proton", kind="bfgs", op="solve", n=77373, k=100, rows=0, nnz_row=0.0),
        dict(name="solve_vmat", kind="bfgs", op="solve", n=13425, k=33, rows=68618, nnz_row=134.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["rt", "rt", "rt", "dense", "bfgs"])
    if kind == "dense":
        n = int(_log(rng, 16, 700))
        return dict(kind="dense", op="dir", n=n, m=int(n * rng.uniform(1.0, 2.0)), eta=1e-12)
    if kind == "bfgs":
        if rng.random() < 0.5:
            return dict(kind="bfgs", op="solve", n=int(_log(rng, 2000, 77000)), k=rng.randint(4, 100), rows=0, nnz_row=0.0)
        n = int(_log(rng, 4000, 13425))   # the VMAT shape scaled down
        return dict(kind="bfgs", op="solve", n=n, k=rng.randint(20, 33), rows=int(n * rng.uniform(4.6, 5.1)),
                    nnz_row=0.01 * n)
    op = rng.choice(["solve", "solve", "serve", "batch", "dir", "apply", "resid"])
    n = int(_log(rng, 1100, 20000 if op == "batch" else 50000))
    c = dict(kind="rt", op=op, n=n, nnz_row=min(250.0, max(4.0, rng.uniform(0.002, 0.01) * n)), organ=rng.uniform(0.05, 0.125),
             storage="f64")
    if op == "batch":
        c["count"] = rng.randint(2, 12)
    if op in ("solve", "serve", "batch"):
        c["storage"] = rng.choice(["f64", "f32", "bf16"]) if n < 20000 else "f64"
    if op == "dir":
        c["storage"] = rng.choice(["f64", "f64", "f32", "bf16", "fp8"]) if n < 20000 else "f64"
        c["eta"] = 1e-13 if c["storage"] == "f64" else 1e-12
    return c


# ------------------------------------------------------------------------------------ inputs

class _Draw:
    """Draws of one seed, on the GPU, in float64."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def uniform(self, lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=self.g, device="cuda", dtype=torch.float64)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device="cuda", dtype=torch.float64)


def _bands(d, rows, n, nnz_row):
    """CSR structure of banded rows: about nnz_row entries a row in one to four contiguous bands,
    the first near the diagonal (neighbouring rows overlap), the others anywhere."""
    dev = "cuda"
    p = nnz_row / n
    k = (nnz_row + math.sqrt(nnz_row * (1 - p)) * d.normal(rows)).round().clamp(1, n).long()
    nb = 1 + (d.uniform(0, 1, rows, 3) < 0.5).sum(1)
    u = d.uniform(0, 1, rows, 4)
    u[torch.arange(4, device=dev)[None, :] >= nb[:, None]] = 0.0
    ln = torch.floor(u / u.sum(1, keepdim=True) * k[:, None]).long()
    ln[:, 0] += k - ln.sum(1)
    centre = torch.empty(rows, 4, device=dev, dtype=torch.float64)
    centre[:, 0] = (torch.arange(rows, device=dev) + 0.5) * (n / rows) + 0.02 * n * d.normal(rows)
    centre[:, 1:] = d.uniform(0, n, rows, 3)
    st = (centre - ln / 2.0).round().long()
    st = torch.minimum(st.clamp(min=0), (n - ln).clamp(min=0))
    order = torch.argsort(torch.where(ln > 0, st, n + 1), dim=1, stable=True)
    st, en = st.gather(1, order), (st + ln).gather(1, order)
    en = torch.where(en > st, en, torch.zeros_like(en))   # an unused band ends before every other begins
    prev = torch.cat([torch.zeros(rows, 1, device=dev, dtype=torch.long), torch.cummax(en, 1).values[:, :-1]], 1)
    st = torch.maximum(st, prev)
    ln = (en - st).clamp(min=0)
    ptr = torch.zeros(rows + 1, device=dev, dtype=torch.long)
    ptr[1:] = torch.cumsum(ln.sum(1), 0)
    ln, st = ln.reshape(-1), st.reshape(-1)
    first = torch.cumsum(ln, 0) - ln
    total = int(ln.sum())
    idx = torch.repeat_interleave((st - first).int(), ln) + torch.arange(total, device=dev, dtype=torch.int32)
    return ptr, idx


def _row_of(ptr):
    return torch.repeat_interleave(torch.arange(ptr.numel() - 1, device="cuda"), ptr[1:] - ptr[:-1])


def _sum_into(size, where, v):
    """sum of v by index, in integers of 2^-30 (the same bits in any order)."""
    s = torch.zeros(size, device="cuda", dtype=torch.int64)
    s.index_add_(0, where, (v * 2.0**30).round().long())
    return s.double() * 2.0**-30


def _problem(case, seed):
    """The QP's arrays (device tensors; the dense QP's on the host)."""
    d = _Draw(seed)
    n = case["n"]
    if case["kind"] == "dense":
        m = case["m"]
        rng = np.random.default_rng(seed)
        A = rng.normal(0.0, 1.0 / math.sqrt(n), size=(m, n))
        Q = np.linalg.qr(rng.normal(size=(n, n)))[0]
        H = (Q * 10.0 ** rng.uniform(-3.0, 2.0, size=n)[None, :]) @ Q.T
        return dict(n=n, m=m, H=0.5 * (H + H.T), A=A, c=rng.normal(size=n), b=A.sum(1) + rng.uniform(0.1, 1.0, size=m),
                    l=np.zeros(n), u=np.full(n, 10.0))
    p = dict(n=n)
    if case["kind"] == "rt":
        V = 4 * n
        m = max(1, int(V * case["organ"]))
        ptr, idx = _bands(d, V, n, case["nnz_row"])
        val = torch.exp(d.normal(idx.numel()))
        w = d.uniform(0.1, 10.0, V)
        voxel = torch.randperm(V, generator=d.g, device="cuda")
        presc = torch.zeros(V, device="cuda", dtype=torch.float64)
        presc[voxel[:int(0.3 * V)]] = 1.0
        c = -_sum_into(n, idx, val * (w * presc)[_row_of(ptr)])
        p.update(m=m, F=(ptr, idx, val), f_w=w, h0=torch.full((n,), 1e-4, device="cuda", dtype=torch.float64), c=c,
                 a_rows=voxel[int(0.3 * V):][:m].sort().values.int(), b=torch.full((m,), 0.6, device="cuda", dtype=torch.float64),
                 l=torch.zeros(n, device="cuda", dtype=torch.float64), u=torch.full((n,), 5.0, device="cuda", dtype=torch.float64))
        return p
    # quasi-Newton Hessian: k BFGS updates of diag(h0) from pairs (s, y = lam o s)
    k, m = case["k"], case["rows"]
    h0 = d.uniform(0.5, 2.0, n)
    lam = 10.0 ** d.uniform(-2.0, 2.0, n)
    U = torch.zeros(n, 2 * k, device="cuda", dtype=torch.float64)
    uw = torch.zeros(2 * k, device="cuda", dtype=torch.float64)
    for i in range(k):
        s = d.normal(n) / math.sqrt(n)
        hs = h0 * s + U[:, :2 * i] @ (uw[:2 * i] * (U[:, :2 * i].T @ s))
        U[:, 2 * i], U[:, 2 * i + 1] = hs, lam * s
        uw[2 * i], uw[2 * i + 1] = -1.0 / (s @ hs), 1.0 / (s @ (lam * s))
    xt = d.uniform(0.5, 1.5, n)   # the objective pulls towards a plan xt
    c = 0.1 * d.normal(n) - (h0 * xt + U @ (uw * (U.T @ xt))) if m else d.normal(n)
    p.update(m=m, h0=h0, U=U, u_w=uw, c=c, l=torch.zeros(n, device="cuda", dtype=torch.float64),
             u=torch.full((n,), math.inf, device="cuda", dtype=torch.float64))
    if m:
        ptr, idx = _bands(d, m, n, case["nnz_row"])
        row = _row_of(ptr)
        val = torch.exp(d.normal(idx.numel()))
        g1 = _sum_into(m, row, val)
        upper = torch.arange(m, device="cuda") < int(0.77 * m)   # upper rows, then negated lower rows
        p.update(A=(ptr, idx, torch.where(upper[row], val, -val)), b=torch.where(upper, 1.2 * g1, -0.8 * g1))
    return p


def _point(p, seed):
    """A strictly interior point: x between its bounds, log-normal slacks and multipliers."""
    rng = np.random.default_rng([seed, 7])
    n, m = p["n"], p["m"]
    hi = 10.0 if p.get("H") is not None else 5.0
    one = not np.isfinite(float(p["u"][0]))
    return dict(x=hi * rng.uniform(0.05, 0.95, n), s=np.exp(rng.normal(0.0, 0.5, m)), y=np.exp(rng.normal(0.0, 0.5, m)),
                zl=np.exp(rng.normal(0.0, 0.5, n)), zu=np.zeros(n) if one else np.exp(rng.normal(0.0, 0.5, n)), mu=0.1)


def _load(case, p):
    if case["kind"] == "dense":
        return ipm.Solver(tol_kkt=1e-8).set_qp_dense(p["H"], p["c"], p["A"], p["b"], p["l"], p["u"])
    s = ipm.Solver(storage=case.get("storage", "f64"))
    return s.set_qp(p["n"], p["m"], p["c"], p.get("b"), p["l"], p["u"], h0=p["h0"], F=p.get("F"), f_w=p.get("f_w"),
                    a_rows=p.get("a_rows"), A=p.get("A"), U=p.get("U"), u_w=p.get("u_w"))


def prepare(case, seed):
    state = dict(op=case["op"], eta=case.get("eta", 0.0))
    if case["op"] == "batch":
        members = []
        for i in range(case["count"]):
            n = int(case["n"] * (i + 1.5) / (case["count"] + 0.5))   # from a fraction of n up to n, uneven
            c = dict(case, n=n, nnz_row=max(3.0, case["nnz_row"] * n / case["n"]))
            members.append(_load(c, _problem(c, 1000 * seed + i)))
        state.update(solvers=members, batch=ipm.Batch(members))
        return state
    p = _problem(case, seed)
    s = state["solver"] = _load(case, p)
    rng = np.random.default_rng([seed, 9])
    if case["op"] in ("dir", "apply", "resid"):
        q = _point(p, seed)
        s.set_iterate(q["x"], q["s"], q["y"], q["zl"], q["zu"], q["mu"])
    if case["op"] == "apply":
        state["v"] = rng.normal(size=p["n"])
    if case["op"] == "serve":
        state["f_w"] = p["f_w"].cpu().numpy() * (1.0 + 0.01 * rng.uniform(-1.0, 1.0, p["f_w"].numel()))
        state["c"] = p["c"].cpu().numpy() * (1.0 + 0.01 * rng.normal(size=p["n"]))
    return state


def _result(s):
    out = s.get()
    return {k: out[k] for k in ("x", "y", "zl", "zu", "s")}


def run(state):
    if state["op"] == "batch":
        state["batch"].solve()
        return [_result(s) for s in state["solvers"]]
    s = state["solver"]
    if state["op"] == "serve":
        s.update_costs(f_w=state["f_w"], c=state["c"])
    if state["op"] in ("solve", "serve"):
        s.solve()
        return _result(s)
    if state["op"] == "apply":
        return s.apply_kkt(state["v"])
    if state["op"] == "resid":
        return s.residuals()
    out = s.newton_direction(state["eta"])
    return {k: out[k] for k in ("dx", "ds", "dy", "dzl", "dzu")}


def work(case):
    """One reading of the matrices (each entry a value and an index) and of every vector the
    call takes, one writing of those it returns; the operations of one pass over the
    matrices for a residual, one operator application otherwise."""
    if case["op"] == "batch":
        parts = [work(dict(case, op="solve", n=n, nnz_row=max(3.0, case["nnz_row"] * n / case["n"])))
                 for n in (int(case["n"] * (i + 1.5) / (case["count"] + 0.5)) for i in range(case["count"]))]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    n = case["n"]
    if case["kind"] == "dense":
        m = case["m"]
        mat, nnz = 8 * n * (n + m), n * n + 2 * n * m
    elif case["kind"] == "rt":
        nnz = 4 * n * case["nnz_row"]
        mat, m, nnz = 12 * nnz + 48 * n, int(4 * n * case["organ"]), 2 * nnz
    else:
        m = case["rows"]
        nnz = m * case["nnz_row"]
        mat, nnz = 12 * nnz + 8 * m + 16 * n * case["k"], 2 * nnz + 4 * n * case["k"]
    if case["op"] == "apply":
        vec = 8 * (6 * n + 2 * m)
    else:
        vec = 8 * (10 * n + 5 * m)
    return {"bytes": mat + vec, "flops": 2 * nnz}


# ------------------------------------------------------------------------------------ exact

class _Csr:
    """v -> M v and v -> M^T v of a CSR matrix in float64 with torch."""

    def __init__(self, ptr, idx, val, n):
        rows = ptr.numel() - 1
        self.a = torch.sparse_csr_tensor(ptr, idx.long(), val, size=(rows, n))
        at = torch.argsort(idx, stable=True)
        tp = torch.zeros(n + 1, device="cuda", dtype=torch.long)
        tp[1:] = torch.cumsum(torch.bincount(idx, minlength=n), 0)
        self.val, self.idx, self.row = val, idx.long(), _row_of(ptr)
        self.at = torch.sparse_csr_tensor(tp, self.row[at], val[at], size=(n, rows))

    def mv(self, v):
        return self.a @ v

    def tmv(self, v):
        return self.at @ v

    def diag(self, w):   # diag(M^T diag(w) M)
        return torch.zeros(self.a.shape[1], device="cuda", dtype=torch.float64).index_add_(
            0, self.idx, self.val * self.val * w[self.row])


def exact(case, seed):
    if case["op"] not in ("dir", "apply", "resid"):
        return None   # a whole solve ends within a tolerance of the optimum
    p = _problem(case, seed)
    q = {k: torch.as_tensor(v, device="cuda") if isinstance(v, np.ndarray) else v for k, v in _point(p, seed).items()}
    n, m, mu = p["n"], p["m"], q["mu"]
    dev = {k: torch.as_tensor(p[k], device="cuda") for k in ("c", "b", "l", "u") if p.get(k) is not None}
    if case["kind"] == "dense":
        H, A = torch.as_tensor(p["H"], device="cuda"), torch.as_tensor(p["A"], device="cuda")
        hv, hd = (lambda v: H @ v), H.diagonal()
        av, atv, ad = (lambda v: A @ v), (lambda v: A.T @ v), (lambda w: (A * A).T @ w)
    elif case["kind"] == "rt":
        D, rows = _Csr(*p["F"], n), p["a_rows"].long()

        def on_rows(v):
            t = torch.zeros(p["f_w"].numel(), device="cuda", dtype=torch.float64)
            t[rows] = v
            return t
        hv, hd = (lambda v: D.tmv(p["f_w"] * D.mv(v)) + p["h0"] * v), D.diag(p["f_w"]) + p["h0"]
        av, atv, ad = (lambda v: D.mv(v)[rows]), (lambda v: D.tmv(on_rows(v))), (lambda w: D.diag(on_rows(w)))
    else:
        U, uw = p["U"], p["u_w"]
        hv, hd = (lambda v: p["h0"] * v + U @ (uw * (U.T @ v))), p["h0"] + (U * U) @ uw
        if m:
            C = _Csr(*p["A"], n)
            av, atv, ad = C.mv, C.tmv, C.diag
        else:
            av, atv, ad = (lambda v: v[:0]), (lambda w: torch.zeros_like(dev["c"])), (lambda w: torch.zeros_like(dev["c"]))
    b = dev["b"] if m else dev["c"][:0]
    up = torch.isfinite(dev["u"])
    theta = q["y"] / q["s"]
    tl, tu = q["x"] - dev["l"], torch.where(up, dev["u"] - q["x"], 1.0)
    sigma = q["zl"] / tl + q["zu"] / tu

    def kv(v):
        return hv(v) + atv(theta * av(v)) + sigma * v
    if case["op"] == "apply":
        v = torch.as_tensor(np.random.default_rng([seed, 9]).normal(size=n), device="cuda")
        return kv(v).cpu().numpy()
    x, c = q["x"], dev["c"]
    hx, aty, ax = hv(x), atv(q["y"]), av(x)
    rd, rp, rs = hx + c + aty - q["zl"] + q["zu"], ax + q["s"] - b, q["s"] * q["y"] - mu
    rl, ru = tl * q["zl"] - mu, torch.where(up, tu * q["zu"] - mu, 0.0)

    def top(v):
        return float(v.abs().max()) if v.numel() else 0.0
    if case["op"] == "resid":
        pobj = float(0.5 * (x @ hx) + c @ x)
        dobj = float(-0.5 * (x @ hx) - b @ q["y"] + dev["l"] @ q["zl"] - torch.where(up, dev["u"] * q["zu"], 0.0).sum())
        pr = max(0.0, float((ax - b).max()), float((-tl).max()), float(torch.where(up, -tu, -1.0).max())) / (1 + top(b))
        du = top(rd) / (1 + max(top(c), top(hx), top(aty)))
        gap = abs(pobj - dobj) / (1 + abs(pobj) + abs(dobj))
        vec = dict(rd=rd, rp=rp, rs=rs, rl=rl, ru=ru)
        return dict({k: v.cpu().numpy() for k, v in vec.items()}, rel_kkt=max(pr, du, gap), primal=pr, dual=du, gap=gap)
    rhs = -rd - rl / tl + ru / tu - atv(theta * rp - rs / q["s"])
    if n <= 3000:
        K = torch.stack([kv(e) for e in torch.eye(n, device="cuda", dtype=torch.float64)], 1)
        f = torch.linalg.cholesky(0.5 * (K + K.T))
        dx = torch.zeros_like(x)
        for _ in range(3):
            dx = dx + torch.cholesky_solve((rhs - kv(dx))[:, None], f)[:, 0]
    else:
        # Jacobi PCG, restarted on the true residual until that is at rounding level
        minv, dx = 1.0 / (hd + ad(theta) + sigma), torch.zeros_like(x)
        goal, spent = 3e-15 * float(rhs.norm()), 0
        for _ in range(6):
            r = rhs - kv(dx)
            start = float(r.norm())
            if start <= 10 * goal:
                break
            z = minv * r
            v, rz, e = z.clone(), r @ z, torch.zeros_like(x)
            for it in range(4000):
                w = kv(v)
                al = rz / (v @ w)
                e, r = e + al * v, r - al * w
                z = minv * r
                new = r @ z
                v, rz = z + (new / rz) * v, new
                if it % 25 == 24 and float(r.norm()) <= max(goal, 1e-9 * start):
                    break
            dx, spent = dx + e, spent + it
            if spent > 6000:
                return None
    adx = av(dx)
    out = dict(dx=dx, ds=-rp - adx, dy=theta * (adx + rp) - rs / q["s"], dzl=(-rl - q["zl"] * dx) / tl,
               dzu=torch.where(up, (-ru + q["zu"] * dx) / tu, 0.0))
    return {k: v.cpu().numpy() for k, v in out.items()}
