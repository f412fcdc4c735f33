"""The dots of an FP32 or BF16 basis in the fused cycles: a lane's products are FP32, what the lanes,
warps and blocks add up is kept beyond FP32 (double-FP32 pairs), as in the kernels of one phase
each (FP64)."""
import numpy as np
import pytest

from helpers import gpu_solver_from_oracle, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("kind", ["dia", "csr"])
@pytest.mark.parametrize("ortho,prec", [(0, 1), (0, 2), (2, 1)])
def test_sums_over_lanes(orc, ortho, prec, kind, batch):
    """One step on a diagonal matrix from b = 1, whose result is b (sum d) / (sum d^2).  Four rows
    per lane sum to +-2^22 and a multiple of 1/2, exact in FP32; the large parts cancel between
    odd and even lanes and 128 is left, which FP32 sums over the lanes miss by some 8.  All other
    quantities are exact in FP32 (|b| = 16, the projection d - 1/2), but for the norm: 1e-6."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_04051_gb300 as G
    from paper_1906_04051_gb300 import build as B
    B.build()
    n, lanes = 256, 64
    rng = np.random.default_rng(8)
    half = rng.integers(-400, 400, lanes)
    half[-1] += 256 - half.sum()
    d = np.ones(n)
    sign = np.where(np.arange(lanes) % 2, -1.0, 1.0)
    d[0::4] = sign * 2.0 ** 22
    d[1::4] = 0.5 * half
    d[2::4] = 1.0
    d[3::4] = -1.0
    assert d.sum() == 128.0
    rowptr, col, val = np.arange(n + 1), np.arange(n), d
    if kind == "csr":  # zeros all over: no diagonals to store
        other = (np.arange(n) + rng.integers(1, n, n)) % n
        col = np.sort(np.stack([np.arange(n), other], 1), 1)
        val = np.where(col == np.arange(n)[:, None], d[:, None], 0.0).ravel()
        rowptr, col = 2 * rowptr, col.ravel()
    s = gpu_solver_from_oracle(G, orc.CSR(rowptr, col, val), deflation_mode=G.DEFL_NONE, ortho=ortho,
                               precision=prec, fixed_iterations=True)
    assert (s.layout()["ndiag"] > 0) == (kind == "dia")
    b = to_dev(np.ones(n))
    if batch:
        xs, infos, _ = G.batch_solve([s], [b], m=20, tol=0.0, maxit=1)  # (in a cluster)
        x, info = xs[0], infos[0]
        assert s.profile()["arnoldi"][1] > 0
    else:
        x, info = s.solve(b, m=1, tol=0.0, maxit=1)
    assert info["iters"] == 1
    want = 128.0 / np.dot(d, d)
    assert np.abs(x.cpu().numpy() / want - 1.0).max() <= 1e-6
