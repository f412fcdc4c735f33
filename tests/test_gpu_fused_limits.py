"""The sizes up to which a restart cycle runs as one kernel (fused_rows, csrc/fused_fp64.cu), on both
sides of its lines for operators whose SpMV weighs most: 27 diagonals, and long CSR rows with
columns all over the vector (beside the same rows in an order that keeps neighbours together)."""
import itertools

import numpy as np
import pytest

from helpers import gpu_solver_from_oracle, relerr, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _stencil27(orc, n, order):
    """27 neighbours on n^3 nodes; order: None, or the node that each row stands for"""
    rng = np.random.default_rng(n)
    N = n ** 3
    ijk = np.stack(np.unravel_index(np.arange(N), (n, n, n)))
    cols = np.empty((N, 27), dtype=np.int64)
    for q, o in enumerate(itertools.product((-1, 0, 1), repeat=3)):
        nb = ijk + np.array(o)[:, None]
        ok = ((nb >= 0) & (nb < n)).all(0)
        cols[:, q] = np.where(ok, (nb[0] * n + nb[1]) * n + nb[2], N)
    if order is not None:
        inv = np.append(np.argsort(order), N)
        cols = np.sort(inv[cols[order]], 1)
    val = rng.uniform(-0.6, 0.4, cols.shape)
    val[cols == np.arange(N)[:, None]] = 16.0
    there = cols < N
    rowptr = np.concatenate([[0], np.cumsum(there.sum(1))])
    return orc.CSR(rowptr, cols[there], val[there]), rng.standard_normal(N)


# (steps in FP32: 6 x 2^-24 x the condition of the projected problem, below 100: 1e-4)
@pytest.mark.parametrize("n,order,ortho,prec,fused", [
    (97, None, 0, 1, True), (98, None, 0, 1, False),
    (57, "random", 0, 0, True), (58, "random", 0, 0, False), (58, "random", 2, 0, False),
    (58, "tiles", 0, 0, True), (58, "tiles", 2, 1, True)])
def test_both_sides_of_the_lines(orc, n, order, ortho, prec, fused):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04051_gb300 as G
    from paper_1906_04051_gb300 import build as B
    B.build()
    perm = None
    if order:
        perm = np.random.default_rng(1).permutation(n ** 3)
        if order == "tiles":
            t = np.stack(np.unravel_index(perm, (n, n, n))) // 8
            perm = perm[np.argsort((t[0] * 100 + t[1]) * 100 + t[2], kind="stable")]
    A, b = _stencil27(orc, n, perm)
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, ortho=ortho, precision=prec,
                               fixed_iterations=True)
    xg, ig = s.solve(to_dev(b), m=6, tol=0.0, maxit=6)
    assert ig["iters"] == 6
    assert (s.profile()["arnoldi"][1] > 0) == fused
    xo, _ = orc.gmres(A, b, m=6, tol=0.0, maxit=6, fixed_iterations=True,
                      **({"ortho": orc.MGS} if ortho else {}))
    assert relerr(xg.cpu().numpy(), xo) <= (1e-9 if prec == 0 else 1e-4)


# GMRES(1) in FP64 with CGS2 runs its cycles as phases, GMRES(2) fused; a batch as clusters_pay says
@pytest.mark.parametrize("m", [1, 2])
def test_shortest_restarts(orc, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04051_gb300 as G
    from paper_1906_04051_gb300 import build as B
    B.build()
    A, b = _stencil27(orc, 12, None)
    s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, fixed_iterations=True)
    xo, _ = orc.gmres(A, b, m=m, tol=0.0, maxit=8, fixed_iterations=True)
    xg, ig = s.solve(to_dev(b), m=m, tol=0.0, maxit=8)
    assert ig["iters"] == 8 and (s.profile()["arnoldi"][1] > 0) == (m > 1)
    assert relerr(xg.cpu().numpy(), xo) <= 1e-9
    xs, infos, _ = G.batch_solve([s], [to_dev(b)], m=m, tol=0.0, maxit=8)
    assert infos[0]["iters"] == 8
    assert relerr(xs[0].cpu().numpy(), xo) <= 1e-9
