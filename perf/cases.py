"""Measured cases of the solver library: what a user's program has it do, through the package's
public entry points (Solver, batch_solve, q1_solve, q2_bratu_assemble, bratu_newton).

listed() names the cases, draw(rng) gives more of the same ranges, prepare(case, seed) makes what
a program has in hand before the call, run(state) is one pass, work(case) the bytes and
operations a pass cannot do without, exact(case, seed) the same result from plain torch in
64 bits (its own assembly and its own GMRES).

The matrices are the two finite-element families of the library: bilinear Q1
convection-diffusion on an n x n mesh of the unit square (lognormal coefficient, Dirichlet
rows) and the 3-D Bratu problem on n^3 27-node hexahedra.  Fixed-step cases follow the
fixed-iteration protocol (a given number of Arnoldi steps, no convergence test); the others
solve to a tolerance at which the solution itself is pinned down.
"""
import math

import numpy as np
import torch

import paper_1906_04051_gb300 as G

F64 = torch.float64
DEV = "cuda"
ORTHO = {"cgs2": G.ORTHO_CGS2, "lowsync": G.ORTHO_MGS_LOWSYNC}
PREC = {"fp64": G.FP64, "fp32": G.FP32_INNER, "bf16": G.BF16_BASIS}


# ---- the cases ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a 4,225-unknown system solved again and again with a kept handle
        # and the library's defaults (CGS2, GMRES(30), 2 x 4 subdomains); launches and
        # latency count
        dict(name="small-n64", kind="solve", n=64, pe=10.0, sigma=0.0, px=2, py=4, m=30,
             ortho="cgs2", prec="fp64", rhs="smooth", steps=0, tol=1e-12, est=330,
             create=False, unstructured=False),
        # the headline system: a new 1M-unknown matrix (create and solve), FP64, one-reduction
        # MGS, 1024 aggregates, six restart cycles
        dict(name="new-n1024-fp64", kind="solve", n=1024, pe=100.0, sigma=0.5, px=32, py=32,
             m=50, ortho="lowsync", prec="fp64", rhs="noise", steps=300, tol=0.0, est=300,
             create=True, unstructured=False),
        # the library's default orthogonalisation on an odd mid-size mesh, new matrix
        dict(name="new-n511-cgs2", kind="solve", n=511, pe=100.0, sigma=0.5, px=16, py=16,
             m=50, ortho="cgs2", prec="fp64", rhs="noise", steps=150, tol=0.0, est=150,
             create=True, unstructured=False),
        # the largest system (4.2M unknowns, few deflation vectors), two GMRES(40) cycles
        dict(name="large-n2048-fp64", kind="solve", n=2048, pe=50.0, sigma=0.5, px=8, py=8,
             m=40, ortho="lowsync", prec="fp64", rhs="noise", steps=80, tol=0.0, est=80,
             create=False, unstructured=False),
        # mixed precision: FP32 inner cycles refined in FP64 to a true 1e-12
        dict(name="mixed-n1024-fp32", kind="solve", n=1024, pe=100.0, sigma=0.5, px=32, py=32,
             m=50, ortho="lowsync", prec="fp32", rhs="noise", steps=0, tol=1e-12, est=1200,
             create=False, unstructured=False),
        # the same with the Krylov basis stored in BF16
        dict(name="mixed-n601-bf16", kind="solve", n=601, pe=20.0, sigma=0.5, px=18, py=18,
             m=40, ortho="cgs2", prec="bf16", rhs="noise", steps=0, tol=1e-12, est=1000,
             create=False, unstructured=False),
        # a mesh numbered by a partitioner: no diagonals, the general CSR path
        dict(name="unstructured-n487", kind="solve", n=487, pe=40.0, sigma=0.3, px=15, py=15,
             m=40, ortho="cgs2", prec="fp64", rhs="noise", steps=120, tol=0.0, est=120,
             create=False, unstructured=True),
        # 64 Newton linearisations of uneven size, deflated, in one call
        dict(name="batch64-fp64", kind="batch", count=64, nmin=32, nmax=128, pe=20.0, m=30,
             ortho="lowsync", prec="fp64", r=8, maxit=6000, tol=1e-11, est=500),
        # the same kind of batch with FP32 inner cycles, no deflation, default CGS2
        dict(name="batch48-fp32", kind="batch", count=48, nmin=24, nmax=96, pe=20.0, m=30,
             ortho="cgs2", prec="fp32", r=0, maxit=6000, tol=1e-11, est=400),
        # a differentiable solve: forward, adjoint and coefficient gradient (new matrix)
        dict(name="grad-n384", kind="grad", n=384, pe=20.0, sigma=0.3, px=12, py=12, m=50,
             ortho="cgs2", tol=1e-10, est=700),
        # a Newton step of the 3-D Bratu problem: assembly at u, create, two GMRES(50) cycles
        dict(name="bratu-n32", kind="bratu", n=32, m=50, ortho="cgs2", steps=100, est=100),
        # the whole nonlinear solve in one call (adaptive deflation, the driver's defaults)
        dict(name="newton-n10", kind="newton", n=10, m=50, est=250),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "grad", "bratu", "newton"])
    if kind == "batch":
        prec = rng.choice(["fp64", "fp32"])
        nmin = rng.randint(20, 40)
        return dict(kind=kind, count=_log(rng, 6, 48), nmin=nmin,
                    nmax=_log(rng, nmin + 10, 128 if prec == "fp64" else 96),
                    pe=round(rng.uniform(5.0, 20.0), 2), m=rng.choice([30, 40]),
                    ortho=rng.choice(["lowsync", "cgs2"]), prec=prec,
                    r=8 if prec == "fp64" else 0, maxit=6000, tol=1e-11, est=500)
    if kind == "grad":
        n = _log(rng, 48, 384)
        px = max(2, n // 32)
        return dict(kind=kind, n=n, pe=round(rng.uniform(5.0, 25.0), 2), sigma=0.3, px=px, py=px,
                    m=rng.choice([40, 50]), ortho=rng.choice(["cgs2", "lowsync"]), tol=1e-10,
                    est=2 * n)
    if kind == "bratu":
        return dict(kind=kind, n=rng.randint(5, 32), m=rng.choice([30, 50]),
                    ortho=rng.choice(["cgs2", "lowsync"]), steps=rng.randint(60, 100), est=100)
    if kind == "newton":
        return dict(kind=kind, n=rng.randint(4, 10), m=rng.randint(30, 60), est=250)
    prec = rng.choice(["fp64", "fp64", "fp64", "fp32", "bf16"])
    if prec != "fp64":
        n = _log(rng, 100, 900)
        px = max(2, n // 32)
        return dict(kind=kind, n=n, pe=round(rng.uniform(10.0, 100.0), 2), sigma=0.5, px=px, py=px,
                    m=rng.choice([40, 50]), prec=prec,
                    ortho="cgs2" if prec == "bf16" else rng.choice(["cgs2", "lowsync"]),
                    rhs="noise", steps=0, tol=1e-12, est=1000, create=False, unstructured=False)
    n = _log(rng, 40, 1500)
    # aggregates of some 32 x 32 nodes, at most 32 x 32 of them; now and then none at all
    px = min(32, max(2, n // 32))
    px, py = rng.choice([(px, px), (px, px), (0, 0)])
    m = rng.choice([30, 40, 50])
    steps = rng.randint(60, 120)
    un = n <= 600 and rng.random() < 0.25
    return dict(kind=kind, n=n, pe=round(rng.uniform(10.0, 100.0), 2), sigma=0.5, px=px, py=py,
                m=m, ortho=rng.choice(["lowsync", "cgs2"]), prec="fp64", rhs="noise",
                steps=steps, tol=0.0, est=steps, create=rng.random() < 0.4, unstructured=un)


# ---- inputs ------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _smooth(n, g):
    """A smooth random nodal field: low sine modes with normal coefficients."""
    t = torch.arange(n + 1, dtype=F64, device=DEV) / n
    k = torch.arange(1, 5, dtype=F64, device=DEV)
    S = torch.sin(math.pi * k[:, None] * t[None, :])
    a = torch.randn(4, 4, generator=g, dtype=F64, device=DEV) / torch.sqrt(
        k[:, None] ** 2 + k[None, :] ** 2)
    return S.t() @ a @ S  # (j, i)


def _q1_rows(n, kappa, beta, f, u=None):
    """Q1 system by rows: columns and values (N x 9), the entries that exist, and b.
    kappa is (n, n) indexed [ej, ei]; f and u are (n + 1, n + 1) indexed [j, i]."""
    h, np1 = 1.0 / n, n + 1
    S = ((1.0, -1.0), (-1.0, 1.0))
    M = ((1.0 / 3.0, 1.0 / 6.0), (1.0 / 6.0, 1.0 / 3.0))
    D = (-0.5, 0.5)
    V = torch.zeros(9, np1, np1, dtype=F64, device=DEV)
    b = torch.zeros(np1, np1, dtype=F64, device=DEV)
    c0 = slice(1, n)
    for a in (0, 1):
        for bb in (0, 1):
            ke = kappa[1 - bb:n - bb, 1 - a:n - a]
            for c in (0, 1):
                for d in (0, 1):
                    di, dj = c - a, d - bb
                    k1 = S[a][c] * M[bb][d] + M[a][c] * S[bb][d]
                    cc = h * (beta[0] * D[c] * M[bb][d] + beta[1] * M[a][c] * D[d])
                    v = ke * k1 + cc
                    V[(dj + 1) * 3 + di + 1, c0, c0] += v
                    at = (slice(1 + dj, n + dj), slice(1 + di, n + di))
                    b[c0, c0] += h * h * M[a][c] * M[bb][d] * f[at]
                    if u is not None:
                        b[c0, c0] -= v * u[at]
    inner = torch.zeros(np1, np1, dtype=torch.bool, device=DEV)
    inner[c0, c0] = True
    V[4][~inner] = 1.0
    N = np1 * np1
    off = torch.tensor([dj * np1 + di for dj in (-1, 0, 1) for di in (-1, 0, 1)], device=DEV)
    col = torch.arange(N, device=DEV)[:, None] + off[None, :]
    live = inner.reshape(-1, 1).expand(N, 9).clone()
    live[:, 4] = True
    return col, V.reshape(9, N).t().contiguous(), live, b.reshape(-1)


def _csr(col, val, live):
    rowptr = torch.zeros(col.shape[0] + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = torch.cumsum(live.sum(1), 0).to(torch.int32)
    return rowptr, col[live].to(torch.int32), val[live].contiguous()


def _aggregates(n, px, py):
    i = torch.arange(n + 1, device=DEV)
    return ((i * px) // (n + 1))[None, :].add(px * ((i * py) // (n + 1))[:, None]).reshape(-1)


def _q1_system(case, seed):
    """(rowptr, col, val, b, agg or None, r) of a "solve" case."""
    n, g = case["n"], _gen(seed)
    beta = (case["pe"] * math.cos(0.3), case["pe"] * math.sin(0.3))
    kappa = torch.exp(case["sigma"] * torch.randn(n, n, generator=g, dtype=F64, device=DEV))
    if case["rhs"] == "noise":
        f = 2.0 * torch.rand(n + 1, n + 1, generator=g, dtype=F64, device=DEV) - 1.0
    else:
        f = 1.0 + _smooth(n, g)
    col, val, live, b = _q1_rows(n, kappa, beta, f)
    r = case["px"] * case["py"]
    agg = _aggregates(n, case["px"], case["py"]) if r else None
    if case["unstructured"]:
        # a partitioner's numbering: parts of some 1000 nodes in turn, any order inside one
        parts = max(2, n // 32)
        key = _aggregates(n, parts, parts).to(F64) + torch.rand(
            col.shape[0], generator=g, dtype=F64, device=DEV)
        perm = torch.argsort(key)
        inv = torch.empty_like(perm)
        inv[perm] = torch.arange(perm.numel(), device=DEV)
        col, val, live, b = col[perm], val[perm], live[perm], b[perm].contiguous()
        agg = agg[perm] if agg is not None else None
        col = torch.where(live, inv[col.clamp(0, perm.numel() - 1)],
                          torch.full_like(col, perm.numel()))
        col, order = torch.sort(col, dim=1)
        val, live = torch.gather(val, 1, order), torch.gather(live, 1, order)
    rowptr, col, val = _csr(col, val, live)
    return rowptr, col, val, b, agg.to(torch.int32) if agg is not None else None, r


def _batch_systems(case, seed):
    g = _gen(seed)
    lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
    # sizes spread evenly over the logarithm of the range and dealt in a fixed shuffle, so
    # that every seed has the same total work
    k = case["count"]
    order = np.random.RandomState(7).permutation(k)
    sizes = [int(round(math.exp(lo + (hi - lo) * (i + 0.5) / k))) for i in order]
    pes = (1.0 + (case["pe"] - 1.0) * torch.rand(k, generator=g, dtype=F64, device=DEV)).tolist()
    out = []
    for n, pe in zip(sizes, pes):
        u = _smooth(n, g)
        c = 0.25 * (u[:-1, :-1] + u[:-1, 1:] + u[1:, :-1] + u[1:, 1:])
        beta = (pe * math.cos(0.3), pe * math.sin(0.3))
        col, val, live, b = _q1_rows(n, 1.0 + c * c, beta, torch.ones_like(u), u)
        agg = _aggregates(n, 2, 4).to(torch.int32) if case["r"] else None
        out.append((*_csr(col, val, live), b, agg, case["r"]))
    return out


def _grad_inputs(case, seed):
    n, g = case["n"], _gen(seed)
    kappa = torch.exp(case["sigma"] * torch.randn(n * n, generator=g, dtype=F64, device=DEV))
    beta = (case["pe"] * math.cos(0.3), case["pe"] * math.sin(0.3))
    _, _, _, b = _q1_rows(n, torch.ones(n, n, dtype=F64, device=DEV), beta, 1.0 + _smooth(n, g))
    target = 0.1 * _smooth(n, g).reshape(-1).contiguous()
    return kappa, beta, b, target


def _bratu_u(case, seed):
    """A Newton iterate: smooth, zero on the x- and y-faces; and lambda."""
    M, g = 2 * case["n"] + 1, _gen(seed)
    t = torch.arange(M, dtype=F64, device=DEV) / (M - 1)
    s = torch.sin(math.pi * t)
    c = torch.rand(3, generator=g, dtype=F64, device=DEV)
    z = 1.0 + 0.2 * c[0] * torch.cos(math.pi * t) + 0.1 * c[1] * torch.cos(2.0 * math.pi * t)
    u = 0.8 * z[:, None, None] * s[None, :, None] * s[None, None, :]
    return u.reshape(-1).contiguous(), 2.0 + 4.0 * float(c[2])


def _solver(case, sys_):
    rowptr, col, val, _, agg, r = sys_
    return G.Solver(rowptr, col, val, agg, r, precision=PREC[case["prec"]],
                    ortho=ORTHO[case["ortho"]],
                    deflation_mode=G.DEFL_EBP if r else G.DEFL_NONE,
                    fixed_iterations=case.get("steps", 0) > 0)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "solve":
        s["sys"] = _q1_system(case, seed)
        s["solver"] = None if case["create"] else _solver(case, s["sys"])
    elif case["kind"] == "batch":
        s["sys"] = _batch_systems(case, seed)
        s["solvers"] = [_solver(case, q) for q in s["sys"]]
    elif case["kind"] == "grad":
        s["in"] = _grad_inputs(case, seed)
        agg = _aggregates(case["n"], case["px"], case["py"]).to(torch.int32)
        s["setup"] = G.Q1Setup(case["n"], s["in"][1], agg, case["px"] * case["py"], m=case["m"],
                               tol=case["tol"], ortho=ORTHO[case["ortho"]])
    else:
        s["u"], s["lam"] = _bratu_u(case, seed)
    return s


# ---- one pass ----------------------------------------------------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        solver = state["solver"] or _solver(case, state["sys"])
        x, _ = solver.solve(state["sys"][3], m=case["m"], tol=case["tol"],
                            maxit=case["steps"] or 20000)
        if state["solver"] is None:
            solver.close()
        return x
    if case["kind"] == "batch":
        xs, _, _ = G.batch_solve(state["solvers"], [q[3] for q in state["sys"]], m=case["m"],
                                 tol=case["tol"], maxit=case["maxit"])
        return xs
    if case["kind"] == "grad":
        kappa, _, b, target = state["in"]
        kappa, b = kappa.detach().requires_grad_(), b.detach().requires_grad_()
        x = G.q1_solve(kappa, b, state["setup"])
        (x - target).square().sum().backward()
        return {"x": x.detach(), "kappa_grad": kappa.grad, "b_grad": b.grad}
    if case["kind"] == "bratu":
        rowptr, col, val, b = G.q2_bratu_assemble(case["n"], state["lam"], state["u"])
        solver = G.Solver(rowptr, col, val, deflation_mode=G.DEFL_NONE,
                          ortho=ORTHO[case["ortho"]], fixed_iterations=True)
        x, _ = solver.solve(b, m=case["m"], tol=0.0, maxit=case["steps"])
        solver.close()
        return {"rowptr": rowptr, "col": col, "val": val, "b": b, "x": x}
    u, _ = G.bratu_newton(case["n"], state["lam"], state["u"].clone(), m=case["m"])
    return u


# ---- the work of a pass ------------------------------------------------------------------
def work(case):
    """Inputs read once and outputs written once; operations of the steps that the method
    takes (SpMV and, per step with k basis columns, k dot products and k updates; the step
    count of a solve to a tolerance is the case's estimate)."""
    def q1(n, steps, m):
        N, nnz = (n + 1) ** 2, 9 * (n - 1) ** 2 + 4 * n
        return 12.0 * nnz + 4.0 * N + 16.0 * N, steps * (2.0 * nnz + 2.0 * (m + 1) * N)

    kind, est = case["kind"], case["est"]
    if kind == "solve":
        by, fl = q1(case["n"], est, case["m"])
    elif kind == "batch":
        k = case["count"]
        lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
        ns = [int(round(math.exp(lo + (hi - lo) * (i + 0.5) / k))) for i in range(k)]
        by = sum(q1(n, est, case["m"])[0] for n in ns)
        fl = sum(q1(n, est, case["m"])[1] for n in ns)
    elif kind == "grad":
        n = case["n"]
        N = (n + 1) ** 2
        fl = 2.0 * q1(n, est, case["m"])[1]
        by = 8.0 * (2 * n * n + 4 * N) + 4.0 * N
    else:
        M, S = 2 * case["n"] + 1, 8 * case["n"] - 5
        N, nnz = M ** 3, M * (4 * M - 4) + S * S * (S + 6)
        fl = est * (2.0 * nnz + 2.0 * (case["m"] + 1) * N)
        by = 12.0 * nnz + 4.0 * N + 24.0 * N if kind == "bratu" else 16.0 * N
    return {"bytes": by, "flops": fl}


# ---- the same in plain torch, 64 bits ------------------------------------------------------
def _sparse(rowptr, col, val):
    n = rowptr.numel() - 1
    return torch.sparse_csr_tensor(rowptr.to(torch.int64), col.to(torch.int64), val, (n, n))


def _gmres(A, b, m, steps=None, agg=None, r=0):
    """Restarted GMRES(m) from x = 0, right-preconditioned by I + U (|mu| T^-1 - I) U^T (U the
    normalised aggregate indicators, T = U^T A U, mu from the Ritz values of the first,
    unpreconditioned cycle).  steps: exactly that many; None: the solution itself, by long
    unpreconditioned cycles until the residual stops falling."""
    if steps is None:
        m, r = 150, 0
    n = b.numel()
    if r:
        agg = agg.to(torch.int64)
        us = torch.bincount(agg, minlength=r).to(F64).rsqrt()
        rows = torch.repeat_interleave(torch.arange(n, device=DEV), A.crow_indices().diff())
        T = torch.zeros(r * r, dtype=F64, device=DEV).index_add_(
            0, agg[rows] * r + agg[A.col_indices()], A.values()).reshape(r, r)
        Ti = torch.linalg.inv(T * us[:, None] * us[None, :])
    mu = None

    def prec(v):
        if not r or mu is None:
            return v
        c = us * torch.zeros(r, dtype=F64, device=DEV).index_add_(0, agg, v)
        return v + (us * (mu * (Ti @ c) - c))[agg]

    V = torch.zeros(m + 1, n, dtype=F64, device=DEV)
    x = torch.zeros_like(b)
    res = b.clone()
    beta0 = beta = float(torch.linalg.norm(res))
    done, bad, best = 0, 0, math.inf
    while beta > 0.0:
        kk = m if steps is None else min(m, steps - done)
        if kk <= 0:
            break
        H = torch.zeros(m + 1, m, dtype=F64, device=DEV)
        V[0] = res / beta
        for j in range(kk):
            w = A @ prec(V[j])
            h = V[:j + 1] @ w
            w -= V[:j + 1].t() @ h
            h2 = V[:j + 1] @ w
            w -= V[:j + 1].t() @ h2
            nw = torch.linalg.norm(w)
            H[:j + 1, j] = h + h2
            H[j + 1, j] = nw
            V[j + 1] = w / nw
        Hc = H.cpu().numpy()
        e = np.zeros(kk + 1)
        e[0] = beta
        y = np.linalg.lstsq(Hc[:kk + 1, :kk], e, rcond=None)[0]
        x = x + prec(torch.from_numpy(y).to(DEV) @ V[:kk])
        if mu is None:
            mu = float(np.abs(np.linalg.eigvals(Hc[:kk, :kk])).max())
        res = b - A @ x
        beta = float(torch.linalg.norm(res))
        done += kk
        if steps is None:
            bad = bad + 1 if beta > 0.7 * best else 0
            best = min(best, beta)
            if beta <= 1e-14 * beta0 or (bad >= 3 and beta < 1e-9 * beta0) or done > 9000:
                break
    return x


def _bratu_system(n, lam, u):
    """J(u) and -R(u) from dense element matrices (3 x 3 x 3 Gauss points): rowptr, col,
    val, b, columns ascending, x- and y-face rows replaced by du_i = 0."""
    M, h = 2 * n + 1, 1.0 / n
    xg = torch.tensor([0.5 - math.sqrt(0.15), 0.5, 0.5 + math.sqrt(0.15)], dtype=F64, device=DEV)
    wg = torch.tensor([5.0, 8.0, 5.0], dtype=F64, device=DEV) / 18.0
    P = torch.stack([(1 - xg) * (1 - 2 * xg), 4 * xg * (1 - xg), xg * (2 * xg - 1)], 1)
    D = torch.stack([4 * xg - 3, 4 - 8 * xg, 4 * xg - 1], 1)
    M1, S1 = P.t() @ (wg[:, None] * P), D.t() @ (wg[:, None] * D)

    def kron(a, b_, c):
        return torch.kron(c, torch.kron(b_, a))

    Ke = h * (kron(S1, M1, M1) + kron(M1, S1, M1) + kron(M1, M1, S1))
    Pq = kron(P, P, P)                                    # 27 points x 27 functions
    wq = h ** 3 * kron(wg[:, None], wg[:, None], wg[:, None]).reshape(-1)
    e = torch.arange(n, device=DEV)
    first = ((2 * e[:, None, None] * M + 2 * e[None, :, None]) * M + 2 * e[None, None, :]).reshape(-1)
    a = torch.arange(3, device=DEV)
    loc = ((a[:, None, None] * M + a[None, :, None]) * M + a[None, None, :]).reshape(-1)
    nodes = first[:, None] + loc[None, :]                 # elements x 27
    ue = u[nodes]
    eq = lam * wq * torch.exp(ue @ Pq.t())
    Je = torch.einsum("eq,ql,qm->elm", eq, Pq, Pq) - Ke
    be = ue @ Ke - eq @ Pq
    N = M ** 3
    b = torch.zeros(N, dtype=F64, device=DEV).index_add_(0, nodes.reshape(-1), be.reshape(-1))
    t = torch.arange(M, device=DEV)
    edge = (t == 0) | (t == M - 1)
    face = (edge[None, None, :] | edge[None, :, None]).expand(M, M, M).reshape(-1)
    keep = ~face[nodes][:, :, None].expand(-1, 27, 27).reshape(-1)
    key = (nodes[:, :, None] * N + nodes[:, None, :]).reshape(-1)[keep]
    f = torch.nonzero(face).reshape(-1)
    key, inv = torch.unique(torch.cat([key, f * N + f]), return_inverse=True)
    val = torch.zeros(key.numel(), dtype=F64, device=DEV).index_add_(
        0, inv, torch.cat([Je.reshape(-1)[keep], torch.ones(f.numel(), dtype=F64, device=DEV)]))
    b[f] = 0.0
    rowptr = torch.zeros(N + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(key // N, minlength=N), 0)
    return rowptr, key % N, val, b


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        rowptr, col, val, b, agg, r = _q1_system(case, seed)
        return _gmres(_sparse(rowptr, col, val), b, case["m"], case["steps"] or None, agg, r)
    if kind == "batch":
        return [_gmres(_sparse(*q[:3]), q[3], case["m"]) for q in _batch_systems(case, seed)]
    if kind == "grad":
        n = case["n"]
        kappa, beta, b, target = _grad_inputs(case, seed)
        col, val, live, _ = _q1_rows(n, kappa.reshape(n, n), beta, torch.zeros(
            n + 1, n + 1, dtype=F64, device=DEV))
        rowptr, col, val = _csr(col, val, live)
        A = _sparse(rowptr, col, val)
        rows = torch.repeat_interleave(torch.arange(b.numel(), device=DEV), A.crow_indices().diff())
        At = torch.sparse_coo_tensor(torch.stack([A.col_indices(), rows]), val, A.shape)
        At = At.coalesce().to_sparse_csr()
        agg, r = _aggregates(n, case["px"], case["py"]), case["px"] * case["py"]
        x = _gmres(A, b, case["m"], None, agg, r)
        lam = _gmres(At, 2.0 * (x - target), case["m"], None, agg, r)
        li = lam.reshape(n + 1, n + 1).clone()
        li[0] = li[n] = 0.0
        li[:, 0] = li[:, n] = 0.0
        xs = x.reshape(n + 1, n + 1)
        S, M = ((1.0, -1.0), (-1.0, 1.0)), ((1 / 3, 1 / 6), (1 / 6, 1 / 3))
        gk = torch.zeros(n, n, dtype=F64, device=DEV)
        for a in (0, 1):
            for bb in (0, 1):
                for c in (0, 1):
                    for d in (0, 1):
                        k1 = S[a][c] * M[bb][d] + M[a][c] * S[bb][d]
                        gk -= k1 * li[bb:n + bb, a:n + a] * xs[d:n + d, c:n + c]
        return {"x": x, "kappa_grad": gk.reshape(-1), "b_grad": lam}
    u, lam = _bratu_u(case, seed)
    if kind == "bratu":
        rowptr, col, val, b = _bratu_system(case["n"], lam, u)
        x = _gmres(_sparse(rowptr, col, val), b, case["m"], case["steps"])
        return {"rowptr": None, "col": None, "val": val, "b": b, "x": x}
    for _ in range(12):  # Newton's method with dense solves
        rowptr, col, val, b = _bratu_system(case["n"], lam, u)
        A = _sparse(rowptr, col, val).to_dense()
        du = torch.linalg.solve(A, b)
        u = u + du
        if float(du.abs().max()) <= 1e-13:
            break
    return u
