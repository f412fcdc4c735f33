"""The exchanges of the fused Arnoldi cycles between blocks (csrc/fused.cuh): partial sums and the
tables of the coarse solve that other blocks, or other phases of the same block, must not meet
half-written.  Small systems, where a phase takes the least time, solved again and again: the
sums have a fixed order, so every solve gives the same bits."""
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


# CGS2's two multi-dots of a step: 128 rows per block and few columns, the shortest second pass
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n,m", [(64, 3), (64, 30), (136, 5)])
def test_cgs2_solves_repeat_bitwise(G, orc, n, m, prec):
    p = W.convdiff(n, pe=20.0, sigma=0.5, seed=n, px=2, py=2)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    kw = dict(mu_mode=1, mu_user=4.0, fixed_iterations=True)
    s = gpu_solver_from_oracle(G, A, p.agg, p.r, precision=prec, **kw)
    first = None
    for _ in range(40):
        x, info = s.solve(to_dev(b), m=m, tol=0.0, maxit=4 * m)
        assert info["iters"] == 4 * m
        if first is None:
            first = x.clone()
        assert torch.equal(x, first)
    if prec == 0:
        xo, _ = orc.gmres(A, b, m=m, tol=0.0, maxit=4 * m, defl=orc.Deflation(A, p.agg, p.r), **kw)
        assert relerr(first.cpu().numpy(), xo) <= 1e-9


def _aggregates(n, px, py):
    j, i = np.divmod(np.arange((n + 1) ** 2), n + 1)
    return ((j * py // (n + 1)) * px + i * px // (n + 1)).astype(np.int32)


# the coarse solve of the FP32 one-reduction step over diagonals: more aggregates than rows in a
# block (its vector c then reaches past the rows of w's slice, where its tables used to start),
# as many, and fewer.  20 steps in FP32: 20 x 2^-24 x the condition of the projected problem, some
# 1e-4 at most; a wrong coarse term changes the first digit
@pytest.mark.parametrize("n,px,py", [(64, 16, 16), (64, 16, 8), (64, 43, 3), (40, 13, 12), (90, 8, 8)])
def test_fp32_coarse_tables(G, orc, n, px, py):
    p = W.convdiff(n, pe=20.0, sigma=0.5, seed=n, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    agg, r = _aggregates(n, px, py), px * py
    kw = dict(mu_mode=1, mu_user=4.0)
    s = gpu_solver_from_oracle(G, A, agg, r, ortho=G.ORTHO_MGS_LOWSYNC, precision=G.FP32_INNER,
                               fixed_iterations=True, **kw)
    xo, _ = orc.gmres(A, b, m=20, tol=0.0, maxit=20, defl=orc.Deflation(A, agg, r), ortho=orc.MGS,
                      fixed_iterations=True, **kw)
    first = None
    for _ in range(10):
        x, info = s.solve(to_dev(b), m=20, tol=0.0, maxit=20)
        assert info["iters"] == 20
        first = x.clone() if first is None else first
        assert torch.equal(x, first)
    assert relerr(first.cpu().numpy(), xo) <= 1e-3


# the same in clusters (banded systems only, 16 rows and more a side: one operator form): blocks
# without any rows (4 to 14 units of rows among 16 blocks), with fewer and with more than r
@pytest.mark.parametrize("count,px", [(1, 2), (3, 2), (3, 11), (8, 5), (40, 3)])
def test_fp32_coarse_tables_in_clusters(G, orc, count, px):
    kw = dict(mu_mode=1, mu_user=4.0)
    sys, ss = [], []
    for i in range(count):
        n = [20, 16, 40, 33, 24][i % 5]
        p = W.convdiff(n, pe=15.0, sigma=0.4, seed=60 + i, px=1, py=1)
        A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
        agg = _aggregates(n, px, px)
        sys.append((A, b, agg))
        ss.append(gpu_solver_from_oracle(G, A, agg, px * px, ortho=G.ORTHO_MGS_LOWSYNC,
                                         precision=G.FP32_INNER, fixed_iterations=True, **kw))
        assert ss[-1].layout()["ndiag"] == 9
    bs = [to_dev(b) for _, b, _ in sys]
    first = None
    for _ in range(5):
        xs, infos, _ = G.batch_solve(ss, bs, m=15, tol=0.0, maxit=15)
        assert all(i["iters"] == 15 for i in infos)
        first = [x.clone() for x in xs] if first is None else first
        assert all(torch.equal(x, y) for x, y in zip(xs, first))
    for x, (A, b, agg) in zip(first, sys):
        xo, _ = orc.gmres(A, b, m=15, tol=0.0, maxit=15, defl=orc.Deflation(A, agg, px * px),
                          ortho=orc.MGS, fixed_iterations=True, **kw)
        assert relerr(x.cpu().numpy(), xo) <= 1e-3


# blocks of a cluster without any rows (systems of 2 to 6 units of 128 rows among 8 or 16 blocks)
# add nothing to the dots, from the first step of the first cycle on: against the FP64 oracle, with
# the tolerance of the basis precision (2^-24 or 2^-8 a step, 8 steps, projected problems of
# condition below 100), and bitwise over fresh handles, whose workspaces hold something else
@pytest.mark.parametrize("ortho,prec", [(0, 1), (1, 1), (0, 2)])
@pytest.mark.parametrize("count", [1, 5, 12])
def test_blocks_without_rows(G, orc, count, ortho, prec):
    sys = []
    for i in range(count):
        n = [16, 20, 24][i % 3]
        p = W.convdiff(n, pe=5.0, sigma=0.4, seed=80 + i, px=1, py=1)
        sys.append(orc.q1_assemble(p.n, p.kappa, p.beta, p.f))
    o = G.ORTHO_MGS_LOWSYNC if ortho else G.ORTHO_CGS2
    first = None
    for _ in range(4):
        ss = [gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, ortho=o, precision=prec,
                                     fixed_iterations=True) for A, _ in sys]
        xs, infos, _ = G.batch_solve(ss, [to_dev(b) for _, b in sys], m=8, tol=0.0, maxit=8)
        assert all(i["iters"] == 8 for i in infos)
        first = [x.clone() for x in xs] if first is None else first
        assert all(torch.equal(x, y) for x, y in zip(xs, first))
        for s in ss:
            s.close()
    for x, (A, b) in zip(first, sys):
        xo, _ = orc.gmres(A, b, m=8, tol=0.0, maxit=8, fixed_iterations=True,
                          **({"ortho": orc.MGS} if ortho else {}))
        assert relerr(x.cpu().numpy(), xo) <= (1e-4 if prec == 1 else 0.2)
