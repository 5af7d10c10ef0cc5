"""The FP32 sketch of few points (blocks of 32 rows) at the edges of its tiles, and the factorization
that the Gram kernel's short splits feed.

Bar: the sketch tests' 1e-5 of a column's norm.  (Entries have about 2^-24 (2 + d) |t| log 2 relative
error each, t at most about 20 here where they matter, and sums of at most 2^12 of them add as a
random walk.)"""
import numpy as np
import pytest
import torch

from oracle import krr_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,l", [(1, 1, 1), (31, 3, 2), (32, 8, 31), (33, 16, 33), (63, 5, 127), (64, 6, 64),
                                   (65, 2, 63), (300, 9, 129), (1000, 17, 40), (2049, 4, 110), (4001, 8, 160)])
def test_sketch(n, d, l):
    from paper_1905_10587_gb300.api import KRR
    l = min(l, n)
    rng = np.random.Generator(np.random.PCG64(n + d))
    X = rng.normal(size=(n, d)).astype(np.float32)
    sigma = float(np.sqrt(d))
    Y = KRR().sketch(torch.from_numpy(X).cuda(), sigma, l, seed=11).cpu().numpy()[:, :l]
    ref = O.sketch(X, sigma, O.omega(11, l, n))
    err = np.linalg.norm(Y - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() <= 1e-5


@pytest.mark.parametrize("n,k", [(127, 20), (129, 63), (1023, 64), (1025, 65), (3000, 130)])
def test_gram(n, k):
    from paper_1905_10587_gb300.api import KRR
    rng = np.random.Generator(np.random.PCG64(n + k))
    X = rng.uniform(size=(n, 4)).astype(np.float32) * 3
    S = rng.permutation(n)[:k].astype(np.int32)
    sigma, beta = 0.5, 1e-2
    x = rng.normal(size=(n, 1)).astype(np.float32)
    ctx = KRR(pivot_tol=0.0)
    ctx.build(torch.from_numpy(X).cuda(), sigma, beta, k, anchors=torch.from_numpy(S).cuda())
    z = ctx.apply_precond(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64)
    Xd = X.astype(np.float64)

    def kern(A, B):
        return np.exp(-((A[:, None, :] - B[None, :, :]) ** 2).sum(-1) / (2 * sigma**2))

    C, W = kern(Xd, Xd[S]), kern(Xd[S], Xd[S])
    Kt = C @ np.linalg.solve(W, C.T)
    r = np.linalg.norm(Kt @ z + beta * z - x)
    eta = r / ((np.linalg.norm(Kt, 2) + beta) * np.linalg.norm(z))
    assert eta <= (2 * (k + 5) + k + 2) * 2.0**-24   # test_gpu_parity.py's apply bound
