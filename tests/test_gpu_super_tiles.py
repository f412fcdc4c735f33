"""Fused cycles whose blocks take their rows in more than one super-tile (fused.cuh: w and u_j of one
super-tile at a time are in shared memory, w goes through global memory, dots add up over tiles), and
which path a batch takes: clusters of every size over diagonals, and the phase kernels where a few
large systems would hold up a device of small clusters (clusters_pay, csrc/batch.cu)."""
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


@pytest.fixture(scope="module")
def large(orc):
    p = W.convdiff(1300, pe=50.0, sigma=0.5, seed=17, px=8, py=8)
    return p, *orc.q1_assemble(p.n, p.kappa, p.beta, p.f)


# 1,692,601 rows: 11,135 a block, of which 9,728 without deflation (9,600 with) fit one super-tile;
# wide exponents between the tiles of a block, whose dots are scaled apart
@pytest.mark.parametrize("ortho", [0, 2])
@pytest.mark.parametrize("defl", [False, True])
def test_grid_of_two_super_tiles(G, orc, large, ortho, defl):
    p, A, b = large
    b = b.copy()
    b[(np.arange(b.size) // 1500) % 2 == 1] *= 2.0 ** -40
    kw = dict(mu_mode=1, mu_user=4.0, fixed_iterations=True)
    s = gpu_solver_from_oracle(G, A, p.agg if defl else None, p.r if defl else 0, ortho=ortho,
                               deflation_mode=G.DEFL_EBP if defl else G.DEFL_NONE, **kw)
    xg, ig = s.solve(to_dev(b), m=6, tol=0.0, maxit=9)
    assert ig["iters"] == 9 and s.profile()["arnoldi"][1] == 2
    xo, _ = orc.gmres(A, b, m=6, tol=0.0, maxit=9,
                      **(dict(defl=orc.Deflation(A, p.agg, p.r)) if defl else {}),
                      **({"ortho": orc.MGS} if ortho else {}), **kw)
    assert relerr(xg.cpu().numpy(), xo) <= 1e-9


# clusters of 4 (36 systems): 10,112 rows a block in FP64, 19,776 in FP32 and BF16
@pytest.mark.parametrize("n,ortho,prec", [(200, 0, 0), (200, 2, 0), (280, 0, 1), (280, 2, 1), (280, 0, 2)])
def test_clusters_of_two_super_tiles(G, orc, n, ortho, prec):
    p = W.convdiff(n, pe=20.0, sigma=0.5, seed=n, px=4, py=4)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    kw = dict(mu_mode=1, mu_user=4.0, fixed_iterations=True)
    ss = [gpu_solver_from_oracle(G, A, p.agg, p.r, ortho=ortho, precision=prec, **kw) for _ in range(36)]
    bs = [to_dev(b * (1 + i)) for i in range(36)]
    xs, infos, _ = G.batch_solve(ss, bs, m=5, tol=0.0, maxit=5)
    assert all(s.profile()["arnoldi"][1] > 0 for s in ss)
    xo, _ = orc.gmres(A, b, m=5, tol=0.0, maxit=5, defl=orc.Deflation(A, p.agg, p.r),
                      **({"ortho": orc.MGS} if ortho else {}), **kw)
    for i in (0, 17, 35):  # (5 steps in the basis precision, projected problem of condition < 100)
        assert infos[i]["iters"] == 5
        assert relerr(xs[i].cpu().numpy() / (1 + i), xo) <= (1e-9, 1e-4, 0.2)[prec]


# banded systems only (a mesh of fewer than 16 elements a side goes to CSR): each cluster size (100 of
# these in two waves of clusters with CGS2's longer steps: as phases)
@pytest.mark.parametrize("ortho", [0, 2])
@pytest.mark.parametrize("count", [1, 5, 12, 30, 100])
def test_clusters_over_diagonals(G, orc, count, ortho):
    kw = dict(mu_mode=1, mu_user=4.0, fixed_iterations=True)
    sys, ss = [], []
    for i in range(count):
        p = W.convdiff([16, 33, 24, 40][i % 4], pe=15.0, sigma=0.4, seed=300 + i, px=2, py=1)
        A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
        sys.append((A, b, p))
        ss.append(gpu_solver_from_oracle(G, A, p.agg, p.r, ortho=ortho, **kw))
        assert ss[-1].layout()["ndiag"] == 9
    xs, infos, _ = G.batch_solve(ss, [to_dev(b) for _, b, _ in sys], m=8, tol=0.0, maxit=21)
    assert all(s.profile()["arnoldi"][1] == (0 if count == 100 and ortho == 0 else 3) for s in ss)
    for i in sorted({0, count // 3, count // 2, count - 1}):
        A, b, p = sys[i]
        xo, _ = orc.gmres(A, b, m=8, tol=0.0, maxit=21, defl=orc.Deflation(A, p.agg, p.r),
                          **({"ortho": orc.MGS} if ortho else {}), **kw)
        assert infos[i]["iters"] == 21
        assert relerr(xs[i].cpu().numpy(), xo) <= 1e-9


# 24 systems, one of them of 40,401 rows: alone on a cluster of 4 it would take longer than all
# rows on the whole device as phases; without it, or 36 of its kind, clusters
@pytest.mark.parametrize("big,count,clusters", [(200, 24, False), (60, 24, True), (30, 24, True)])
def test_one_large_system_among_small_ones(G, orc, big, count, clusters):
    sys, ss = [], []
    for i in range(count):
        p = W.convdiff(big if i == 7 else 20, pe=15.0, sigma=0.4, seed=500 + i, px=1, py=1)
        A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
        sys.append((A, b))
        ss.append(gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, fixed_iterations=True))
    xs, infos, _ = G.batch_solve(ss, [to_dev(b) for _, b in sys], m=8, tol=0.0, maxit=21)
    assert all((s.profile()["arnoldi"][1] > 0) == clusters for s in ss)
    for i in (0, 7, count - 1):
        A, b = sys[i]
        xo, _ = orc.gmres(A, b, m=8, tol=0.0, maxit=21, fixed_iterations=True)
        assert infos[i]["iters"] == 21
        assert relerr(xs[i].cpu().numpy(), xo) <= 1e-9
