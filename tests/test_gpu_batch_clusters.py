"""Batched cycles with one thread-block cluster per system (csrc/fused_batch_*.cu): systems of a
few rows (blocks of a cluster without any), numbers of systems on every cluster size and across
their changes as systems finish, and the batches that stay with the phase kernels (operators of
different forms, a system with too many rows)."""
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


def _permuted(orc, A, b, agg, seed):
    """A symmetric permutation, which leaves no diagonals."""
    perm = np.random.default_rng(seed).permutation(A.n)
    inv = np.argsort(perm)
    rows = [sorted(zip(inv[A.col[A.rowptr[i]:A.rowptr[i + 1]]],
                       A.val[A.rowptr[i]:A.rowptr[i + 1]])) for i in perm]
    A = orc.CSR(np.cumsum([0] + [len(q) for q in rows]), np.array([c for q in rows for c, _ in q]),
                np.array([v for q in rows for _, v in q]))
    return A, b[perm], agg[perm]


def _systems(orc, count, kind):
    out = []
    for i in range(count):
        n = [3, 5, 11, 16, 33, 24][i % 6]
        if kind == "big" and i == 0:
            n = 300
        p = W.convdiff(n, pe=15.0, sigma=0.4, seed=900 + i, px=2, py=1)
        A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
        agg = p.agg
        if kind == "csr" or (kind == "mixed" and i == 1):
            A, b, agg = _permuted(orc, A, b, agg, i)
        out.append((A, b, agg, p.r))
    return out


CASES = [(1, "dia"), (13, "dia"), (13, "csr"), (30, "dia"), (60, "csr"), (170, "dia"),
         (5, "mixed"), (3, "big")]


@pytest.mark.parametrize("ortho", [0, 1])
@pytest.mark.parametrize("count,kind", CASES)
def test_fixed_steps_match_oracle(G, orc, count, kind, ortho):
    sys = _systems(orc, count, kind)
    kw = dict(mu_mode=1, mu_user=4.0, fixed_iterations=True)
    o = G.ORTHO_MGS_LOWSYNC if ortho else G.ORTHO_CGS2
    ss = [gpu_solver_from_oracle(G, A, agg, r, ortho=o, **kw) for A, b, agg, r in sys]
    xs, infos, _ = G.batch_solve(ss, [to_dev(b) for _, b, _, _ in sys], m=8, tol=0.0, maxit=21)
    for i in sorted({0, 1 % count, 2 % count, count // 2, count - 2 if count > 1 else 0, count - 1}):
        A, b, agg, r = sys[i]
        if A.n < 60:
            continue  # the Krylov space is exhausted: what remains is rounding
        xo, _ = orc.gmres(A, b, m=8, tol=0.0, maxit=21, defl=orc.Deflation(A, agg, r),
                          **({"ortho": orc.MGS} if ortho else {}), **kw)
        assert infos[i]["iters"] == 21
        assert relerr(xs[i].cpu().numpy(), xo) <= 1e-9


# (the one-reduction form is refused with the BF16 basis)
@pytest.mark.parametrize("ortho,prec", [(0, 0), (0, 1), (0, 2), (1, 0), (1, 1)])
@pytest.mark.parametrize("count,kind", CASES[:-1])
def test_to_tolerance(G, orc, count, kind, ortho, prec):
    sys = _systems(orc, count, kind)
    o = G.ORTHO_MGS_LOWSYNC if ortho else G.ORTHO_CGS2
    ss = [gpu_solver_from_oracle(G, A, agg, r, ortho=o, precision=prec) for A, b, agg, r in sys]
    bs = [to_dev(b) for _, b, _, _ in sys]
    xs, infos, st = G.batch_solve(ss, bs, m=20, tol=1e-10, maxit=20000)
    assert st == 0
    xs = [x.clone() for x in xs]
    for x, (A, b, _, _) in zip(xs, sys):
        assert np.linalg.norm(b - A.matvec(x.cpu().numpy())) <= 1.01e-10 * np.linalg.norm(b)
    xs2, _, _ = G.batch_solve(ss, bs, m=20, tol=1e-10, maxit=20000)
    assert all(torch.equal(x, y) for x, y in zip(xs, xs2))
