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
