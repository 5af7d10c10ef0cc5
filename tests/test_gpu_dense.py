"""The FP64 Cholesky factor and triangular inverses of the preconditioner, through the apply at
anchor counts around the 32-wide diagonal blocks and 16-wide tiles: with every point an anchor the
apply is (K + beta I)^{-1}, and otherwise the Woodbury form against FP64 NumPy.

Bar: the backward error bound of test_gpu_parity.py's apply test, eta = (2 (k + 5) + k + 2) u of
(||K~|| + beta) ||z|| (u = 2^-24): the stored F and the final sums are FP32, so errors of the FP64
factorization well above 1e-8 relative would show."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _backward(n, k, nrhs, seed):
    from paper_1905_10587_gb300.api import KRR
    d, sigma, beta = 4, 0.5, 1e-2
    rng = np.random.Generator(np.random.PCG64(seed))
    X = rng.uniform(size=(n, d)).astype(np.float32) * 2
    S = rng.permutation(n)[:k].astype(np.int32)
    x = rng.normal(size=(n, nrhs)).astype(np.float32)
    ctx = KRR(pivot_tol=0.0)
    ctx.build(torch.from_numpy(X).cuda(), sigma, beta, k, anchors=torch.from_numpy(S).cuda())
    z = ctx.apply_precond(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    Xd = X.astype(np.float64)

    def kern(A, B):
        return np.exp(-((A[:, None, :] - B[None, :, :]) ** 2).sum(-1) / (2 * sigma**2))

    C, W = kern(Xd, Xd[S]), kern(Xd[S], Xd[S])
    Kt = C @ np.linalg.solve(W, C.T)
    r = np.linalg.norm(Kt @ z + beta * z - x, axis=0)
    return (r / ((np.linalg.norm(Kt, 2) + beta) * np.linalg.norm(z, axis=0))).max()


@pytest.mark.parametrize("k", [1, 2, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 97, 130, 257])
def test_apply_at_block_edges(k):
    assert _backward(400, k, 1, k) <= (2 * (k + 5) + k + 2) * 2.0**-24


# every width of a pass over F (1 to 8 columns, then a second pass); few anchors (several row groups
# to a block) and more than 512 (one, and a block to a row of the triangular factors); row counts
# that leave ragged blocks of 16 and 32
@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 6, 7, 8, 9, 16])
@pytest.mark.parametrize("n,k", [(397, 37), (901, 530)])
def test_apply_columns(n, k, nrhs):
    assert _backward(n, k, nrhs, 1000 * k + nrhs) <= (2 * (k + 5) + k + 2) * 2.0**-24
