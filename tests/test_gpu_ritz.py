"""|mu| from the first cycle's Hessenberg matrix by repeated squaring (k_ritz): against the
oracle's eigenvalues for orders 1 to 64, under scaling of A far beyond one, and with a nilpotent
matrix, which has no usable estimate."""
import numpy as np
import pytest

import workloads as W
from helpers import gpu_solver_from_oracle, to_dev

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


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 120, 2.0 ** -90])
@pytest.mark.parametrize("m", [1, 2, 3, 8, 9, 31, 33, 50, 64])
def test_mu_matches_oracle(G, orc, m, scale):
    p = W.convdiff(24, pe=60.0, sigma=0.5, seed=90 + m, px=2, py=2)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    s = gpu_solver_from_oracle(G, orc.CSR(A.rowptr, A.col, A.val * scale), p.agg, p.r)
    _, ig = s.solve(to_dev(b), m=m, tol=1e-30, maxit=m)
    _, io = orc.gmres(A, b, defl=orc.Deflation(A, p.agg, p.r), m=m, tol=1e-30, maxit=m)
    assert ig["mu"] / scale == pytest.approx(io["mu"], rel=1e-10)


def test_nilpotent_matrix_has_no_estimate(G, orc):
    n = 40  # A e_i = e_{i+1}: started from e_0 the Hessenberg matrix is the shift itself
    rowptr = np.concatenate([[0, 0], np.arange(1, n)])
    A = orc.CSR(rowptr, np.arange(n - 1), np.ones(n - 1))
    b = np.zeros(n)
    b[0] = 1.0
    s = gpu_solver_from_oracle(G, A, np.zeros(n, dtype=np.int32), 1)
    with pytest.raises(G.GmresError) as e:
        s.solve(to_dev(b), m=8, tol=1e-8, maxit=100)
    assert e.value.status == -4


# dense upper triangular operators: the powers of H_k grow by 2^1.7 to 2^20 before they settle, where
# squaring alone is off by 1e-10 to 3e-2 (all but the first).  The tolerances are some hundred times
# what relative perturbations of 2e-15 in H_k move the spectral radius by (4e-15, 2e-12, 3e-12, 2e-8)
@pytest.mark.parametrize("n,m,off,tol", [(30, 12, 1.0, 1e-12), (24, 16, 1.0, 2e-10),
                                         (200, 40, 0.2, 3e-10), (40, 33, 0.7, 2e-6)])
def test_strongly_non_normal(G, orc, n, m, off, tol):
    rng = np.random.default_rng(n * 100 + m)
    T = np.triu(rng.standard_normal((n, n)), 1) * off + np.diag(rng.uniform(0.5, 1.5, n))
    b = rng.standard_normal(n)
    A = orc.CSR(np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]),
                np.concatenate([np.arange(i, n) for i in range(n)]),
                np.concatenate([T[i, i:] for i in range(n)]))
    agg = np.zeros(n, dtype=np.int32)
    s = gpu_solver_from_oracle(G, A, agg, 1)
    _, ig = s.solve(to_dev(b), m=m, tol=1e-30, maxit=m)
    _, io = orc.gmres(A, b, defl=orc.Deflation(A, agg, 1), m=m, tol=1e-30, maxit=m)
    assert ig["mu"] == pytest.approx(io["mu"], rel=tol)
    _, ib, _ = G.batch_solve([s], [to_dev(b)], m=m, tol=1e-30, maxit=m)
    assert ib[0]["mu"] == pytest.approx(io["mu"], rel=tol)
