"""The fixed-point dots and column combinations of the FP64 Arnoldi steps (csrc/fixed.cuh): sizes
at the edges of chunks and units, operand ranges that exercise the per-piece exponents, and
exact power-of-two scaling (the integer arithmetic sees the same limbs)."""
import ctypes

import numpy as np
import pytest

import workloads as W
from helpers import gpu_solver_from_oracle, relerr, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04051_gb300 as G
    from paper_1906_04051_gb300 import build as B
    B.build()
    return G


# N = (n + 1)^2: 16 and 121 rows (one unit), 128 +- 16, 256 + 33, 10,201 (ragged units per block)
@pytest.mark.parametrize("n,m", [(3, 9), (10, 33), (11, 20), (16, 64), (100, 37)])
def test_fixed_steps_match_oracle(G, orc, n, m):
    p = W.convdiff(n, pe=30.0, sigma=0.5, seed=7 + n, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    steps = min(2 * m - 1, max(1, (n - 1) ** 2 - 1))
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, fixed_iterations=True,
                               ortho=G.ORTHO_MGS_LOWSYNC)
    xg, ig = s.solve(to_dev(b), m=m, tol=0.0, maxit=steps)
    xo, io = orc.gmres(A, b, m=m, tol=0.0, maxit=steps, fixed_iterations=True, ortho=orc.MGS)
    assert ig["iters"] == io["iters"]
    assert relerr(xg.cpu().numpy(), xo) <= 1e-9


@pytest.mark.parametrize("shift", [-300, 200])
def test_power_of_two_scaling_is_exact(G, orc, shift):
    p = W.convdiff(60, pe=30.0, sigma=0.5, seed=11, px=2, py=2)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    s = gpu_solver_from_oracle(G, A, p.agg, p.r, fixed_iterations=True,
                               ortho=G.ORTHO_MGS_LOWSYNC)
    x1, _ = s.solve(to_dev(b), m=20, tol=0.0, maxit=50)
    x2, _ = s.solve(to_dev(np.ldexp(b, shift)), m=20, tol=0.0, maxit=50)
    assert torch.equal(x1, torch.ldexp(x2, torch.tensor(-shift, device=x2.device)))


# the fused CGS2 cycles: both update passes over a converted basis, operators in diagonals and in
# CSR (short and long rows), every basis precision, row counts at the edges of units and chunks
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n,kind", [(3, "dia"), (15, "dia"), (100, "dia"), (15, "csr"),
                                    (100, "csr"), (2, "long"), (6, "long")])
def test_fused_cgs2_matches_oracle(G, orc, n, kind, prec):
    if kind == "long":
        A, b = orc.q2_bratu_assemble(n, 3.0, np.zeros((2 * n + 1) ** 3))
        agg = (np.arange(A.n) // max(1, A.n // 3)).clip(max=2).astype(np.int32)
        r = 3
    else:
        p = W.convdiff(n, pe=20.0, sigma=0.5, seed=40 + n, px=2, py=1)
        A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
        agg, r = p.agg, p.r
        if kind == "csr":  # a symmetric permutation leaves no diagonals
            perm = np.random.default_rng(n).permutation(A.n)
            inv = np.argsort(perm)
            rows = [sorted(zip(inv[A.col[A.rowptr[i]:A.rowptr[i + 1]]],
                               A.val[A.rowptr[i]:A.rowptr[i + 1]])) for i in perm]
            A = orc.CSR(np.cumsum([0] + [len(q) for q in rows]),
                        np.array([c for q in rows for c, _ in q]),
                        np.array([v for q in rows for _, v in q]))
            b, agg = b[perm], agg[perm]
    steps = min(24, max(1, A.n // 3))
    kw = dict(mu_mode=1, mu_user=4.0)
    if prec == 0:
        s = gpu_solver_from_oracle(G, A, agg, r, fixed_iterations=True, **kw)
        xg, ig = s.solve(to_dev(b), m=10, tol=0.0, maxit=steps)
        xo, _ = orc.gmres(A, b, defl=orc.Deflation(A, agg, r), m=10, tol=0.0, maxit=steps,
                          fixed_iterations=True, **kw)
        assert ig["iters"] == steps
        assert relerr(xg.cpu().numpy(), xo) <= 1e-9
    else:  # FP32 and BF16 inner cycles, refined: the true residual
        s = gpu_solver_from_oracle(G, A, agg, r, precision=prec, **kw)
        xg, ig = s.solve(to_dev(b), m=20, tol=1e-10, maxit=20000)
        assert ig["status"] == 0
        assert np.linalg.norm(b - A.matvec(xg.cpu().numpy())) <= 1.01e-10 * np.linalg.norm(b)


def test_wide_range_of_entries(G, orc):
    """Right-hand side entries over 60 binary orders, one block of rows far below the rest."""
    p = W.convdiff(120, pe=5.0, sigma=0.5, seed=12, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    b = np.ldexp(b, np.random.default_rng(3).integers(-60, 1, b.size))
    b[4000:9000] *= 1e-25
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, fixed_iterations=True,
                               ortho=G.ORTHO_MGS_LOWSYNC)
    xg, _ = s.solve(to_dev(b), m=30, tol=0.0, maxit=60)
    xo, _ = orc.gmres(A, b, m=30, tol=0.0, maxit=60, fixed_iterations=True, ortho=orc.MGS)
    assert relerr(xg.cpu().numpy(), xo) <= 1e-9


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input_is_reported(G, orc, bad):
    p = W.convdiff(40, pe=5.0, sigma=0.5, seed=13, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    A.val[A.rowptr[800]] = bad  # row 800 is an interior row: met in the first SpMV
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, ortho=G.ORTHO_MGS_LOWSYNC)
    with pytest.raises(G.GmresError):
        s.solve(to_dev(b), m=10, tol=1e-8, maxit=50)


# the cycles of an adaptive solve before it has a space are fused ones; its first vectors come from
# their basis in fixed point (or in FP64: double-float dots over diagonals)
@pytest.mark.parametrize("n,kind,ortho,df32", [(9, "dia", 0, 0), (40, "dia", 0, 0), (40, "csr", 0, 0),
                                               (40, "dia", 2, 0), (40, "csr", 2, 0), (40, "dia", 2, 1)])
def test_adaptive_space_from_a_fused_cycle(G, orc, n, kind, ortho, df32):
    p = W.convdiff(n, pe=25.0, sigma=0.5, seed=140, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    if kind == "csr":
        perm = np.random.default_rng(n).permutation(A.n)
        inv = np.argsort(perm)
        rows = [sorted(zip(inv[A.col[A.rowptr[i]:A.rowptr[i + 1]]],
                           A.val[A.rowptr[i]:A.rowptr[i + 1]])) for i in perm]
        A = orc.CSR(np.cumsum([0] + [len(q) for q in rows]),
                    np.array([c for q in rows for c, _ in q]),
                    np.array([v for q in rows for _, v in q]))
        b = b[perm]
    kw = dict(mu_mode=1, mu_user=5.0, rmax=20, fixed_iterations=True)
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_ADAPTIVE, ortho=ortho,
                               dot_arith=G.DOT_DF32 if df32 else G.DOT_FP64, **kw)
    xg, ig = s.solve(to_dev(b), m=15, tol=0.0, maxit=47)
    xo, io = orc.gmres(A, b, m=15, tol=0.0, maxit=47, defl_mode=orc.DEFL_ADAPTIVE,
                       **({"ortho": orc.MGS} if ortho else {}), **kw)
    assert ig["iters"] == io["iters"] == 47
    assert relerr(xg.cpu().numpy(), xo) <= (1e-7 if df32 else 1e-9)


# long rows on both sides of the size up to which their cycles are fused (328,509 and 357,911 rows)
@pytest.mark.parametrize("n", [34, 35])
@pytest.mark.parametrize("ortho", [0, 2])
def test_long_rows_at_the_fused_limit(G, orc, n, ortho):
    A, b = orc.q2_bratu_assemble(n, 3.0, np.zeros((2 * n + 1) ** 3))
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, fixed_iterations=True, ortho=ortho)
    xg, ig = s.solve(to_dev(b), m=6, tol=0.0, maxit=9)
    xo, _ = orc.gmres(A, b, m=6, tol=0.0, maxit=9, fixed_iterations=True,
                      **({"ortho": orc.MGS} if ortho else {}))
    assert ig["iters"] == 9
    assert relerr(xg.cpu().numpy(), xo) <= 1e-9


def _two_blocks(orc, A, b, q, f):
    """diag(A, A) with right-hand sides b and 2^-q b / f."""
    B = orc.CSR(np.concatenate([A.rowptr, A.rowptr[1:] + A.rowptr[-1]]),
                np.concatenate([A.col, A.col + A.n]), np.concatenate([A.val, A.val]))
    return B, np.concatenate([b, np.ldexp(b / f, -q)])


def _permute(orc, A, seed):
    perm = np.random.default_rng(seed).permutation(A.n)
    inv = np.argsort(perm)
    rows = [sorted(zip(inv[A.col[A.rowptr[i]:A.rowptr[i + 1]]],
                       A.val[A.rowptr[i]:A.rowptr[i + 1]])) for i in perm]
    return orc.CSR(np.cumsum([0] + [len(q) for q in rows]), np.array([c for q in rows for c, _ in q]),
                   np.array([v for q in rows for _, v in q])), perm


# An uncoupled block whose right-hand side is 2^-q / f times the other's has a solution in the same
# proportion: all that the blocks share are the projection coefficients.  A basis in fixed point has
# to keep that as FP64 does, however far the block lies below the columns' largest entries, and
# also where its rows start from zeros and grow as the Krylov space spreads ("point": one nonzero
# entry of b).  The bound is what FP64 makes of it: ten times the largest deviation of the
# oracle over three factors f that are not powers of two (3e-16; with an adaptive space 2e-14 to
# 8e-13, since T^-1 amplifies)
@pytest.mark.parametrize("q", [12, 66, 300])
@pytest.mark.parametrize("rhs", ["full", "point"])
@pytest.mark.parametrize("how", ["cgs2", "lowsync", "df32", "csr", "csr-lowsync", "noalloc", "batch",
                                 "batch-lowsync", "adaptive"])
def test_small_uncoupled_block_keeps_its_digits(G, orc, how, rhs, q):
    p = W.convdiff(24, pe=20.0, sigma=0.5, seed=33, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    n = A.n
    if rhs == "point":
        b = np.zeros(n)
        b[n // 2] = 1.0
    bound = 0.0
    for f in (7.0, 1.7, 3.0):
        B, bb = _two_blocks(orc, A, b, q, f)
        xo, _ = orc.gmres(B, bb, m=20, tol=0.0, maxit=60, fixed_iterations=True,
                          **(dict(defl_mode=orc.DEFL_ADAPTIVE, mu_mode=1, mu_user=5.0, rmax=4, ninv=2)
                             if how == "adaptive" else {}))
        bound = max(bound, 10.0 * relerr(f * np.ldexp(xo[n:], q), xo[:n]))
    A, b = B, bb
    perm = np.arange(A.n)
    if how.startswith("csr"):
        A, perm = _permute(orc, A, 3)
    kw = dict(deflation_mode=G.DEFL_NONE, fixed_iterations=True)
    if "lowsync" in how or how == "df32":
        kw["ortho"] = G.ORTHO_MGS_LOWSYNC
    if how == "df32":
        kw["dot_arith"] = G.DOT_DF32
    if how == "adaptive":  # the first cycle is a fused one, whose basis the space comes from
        kw.update(deflation_mode=G.DEFL_ADAPTIVE, mu_mode=1, mu_user=5.0, rmax=4, ninv=2)
    s = gpu_solver_from_oracle(G, A, **kw)
    bd = to_dev(b[perm])
    from paper_1906_04051_gb300 import _native as N
    if how.startswith("batch"):
        xs, infos, _ = G.batch_solve([s], [bd], m=20, tol=0.0, maxit=60)
        x, info = xs[0], infos[0]
    elif how == "noalloc":
        x, info = torch.empty_like(bd), N.gmres_info()
        torch.cuda.synchronize()
        assert N.load().gmres_solve_noalloc(s.handle, bd.data_ptr(), None, 20, 0.0, 60, x.data_ptr(),
                                            ctypes.byref(info)) >= 0
        info = info.as_dict()
    else:
        x, info = s.solve(bd, m=20, tol=0.0, maxit=60)
    assert info["iters"] == 60
    y = np.empty(A.n)
    y[perm] = x.cpu().numpy()
    assert np.linalg.norm(y[:n]) > 0
    assert relerr(3.0 * np.ldexp(y[n:], q), y[:n]) <= bound


# GMRES_DOT_DF32 is for solves with aggregates or without deflation: the undeflated cycles of an
# adaptive or a dense-W solve keep FP64 accuracy, also where floats would underflow
@pytest.mark.parametrize("dense", [False, True])
def test_double_float_dots_not_with_a_dense_space(G, orc, dense):
    p = W.convdiff(40, pe=25.0, sigma=0.5, seed=140, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    kw = dict(rmax=20, ortho=2) if not dense else dict(ortho=2)
    xs = []
    for q, arith in ((-140, G.DOT_DF32), (0, G.DOT_FP64)):
        if dense:
            w = np.linalg.qr(np.random.default_rng(2).standard_normal((A.n, 3)))[0]
            s = G.Solver(to_dev(A.rowptr), to_dev(A.col), to_dev(A.val), w_dense=to_dev(w),
                         fixed_iterations=True, dot_arith=arith, **kw)
        else:
            s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_ADAPTIVE, fixed_iterations=True,
                                       mu_mode=1, mu_user=5.0, dot_arith=arith, **kw)
        x, info = s.solve(to_dev(np.ldexp(b, q)), m=15, tol=0.0, maxit=40)
        assert info["iters"] == 40
        xs.append(np.ldexp(x.cpu().numpy(), -q))
    assert np.array_equal(xs[0], xs[1])
