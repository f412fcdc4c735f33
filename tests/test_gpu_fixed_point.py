"""The fixed-point dots and column combinations of the FP64 Arnoldi steps (csrc/fixed.cuh): sizes
at the edges of chunks and units, operand ranges that exercise the per-piece exponents, and
exact power-of-two scaling (the integer arithmetic sees the same limbs)."""
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
