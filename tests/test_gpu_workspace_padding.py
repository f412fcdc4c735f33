"""The rows between n and the next multiple of 256 of a workspace vector: they are copied with
whole tiles, so they have to hold zeros whatever the memory held before (the fixed-point basis of
a closed handle, say: small negative integers read as NaNs)."""
import numpy as np
import pytest

import workloads as W
from helpers import gpu_solver_from_oracle, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [39, 200])
def test_adaptive_space_after_a_closed_handle(orc, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04051_gb300 as G
    p = W.convdiff(n, pe=10.0, sigma=0.5, seed=21, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    for m in (20, 40, 60, 30, 50):
        s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_NONE, fixed_iterations=True)
        s.solve(to_dev(b), m=m, tol=0.0, maxit=m)
        s.close()
        s = gpu_solver_from_oracle(G, A, deflation_mode=G.DEFL_ADAPTIVE, rmax=6, ninv=2)
        x, info = s.solve(to_dev(b), m=12, tol=1e-3, maxit=400)
        assert info["rel_res_true"] < 1.0
        true = np.linalg.norm(b - A.matvec(x.cpu().numpy())) / np.linalg.norm(b)
        assert true == pytest.approx(info["rel_res_true"], rel=1e-6)
        s.close()


# a solve that meets an infinity says so and leaves nothing behind: the handle's next answer is the one
# it gives without that solve, bit for bit (n + 1 squared is no multiple of 256: there are padding rows)
@pytest.mark.parametrize("prec,ortho", [(0, 0), (0, 2), (1, 0), (1, 2), (2, 0)])
@pytest.mark.parametrize("n", [10, 40])
def test_solve_after_one_that_overflowed(orc, n, prec, ortho):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04051_gb300 as G
    p = W.convdiff(n, pe=10.0, sigma=0.5, seed=23, px=1, py=1)
    A, b = orc.q1_assemble(p.n, p.kappa, p.beta, p.f)
    kw = dict(deflation_mode=G.DEFL_NONE, precision=prec, ortho=ortho, fixed_iterations=True)
    x1, _ = gpu_solver_from_oracle(G, A, **kw).solve(to_dev(b), m=12, tol=0.0, maxit=24)
    s = gpu_solver_from_oracle(G, A, **kw)
    # 1e153: the squares of b's entries are finite, those of A b need not be
    for bad in (b * (1e153 / np.abs(b).max()), np.where(np.arange(b.size) == b.size // 2, np.inf, b)):
        try:
            s.solve(to_dev(bad), m=12, tol=0.0, maxit=24)
        except G.GmresError:
            pass
        x2, _ = s.solve(to_dev(b), m=12, tol=0.0, maxit=24)
        assert torch.equal(x1, x2)
