"""Kernels whose launch overlaps the one before: chains of calls, each on the result of the last,
queued without a host wait and with a wait after every call have to give the same bits."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _data(n, d, r):
    rng = np.random.Generator(np.random.PCG64(n + r))
    X = torch.from_numpy(rng.normal(size=(n, d)).astype(np.float32)).cuda()
    return X, torch.from_numpy(rng.normal(size=(n, r)).astype(np.float32)).cuda()


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,r", [(33, 1), (700, 1), (700, 5), (5003, 1), (5003, 16), (40009, 1)])
def test_chained_products(n, r, precision):
    from paper_1905_10587_gb300.api import KRR
    X, V0 = _data(n, 5, r)
    ctx = KRR(precision=precision)
    out = []
    for wait in (True, False):
        V = V0.clone()
        for _ in range(6):
            V = ctx.kmvm(X, X, V, 2.0, 1e-2)
            V = V / float(n) if wait else V.div_(float(n))
            if wait:
                torch.cuda.synchronize()
        out.append(V.cpu())
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("n,k,r", [(90, 40, 1), (3001, 130, 1), (3001, 130, 8), (25001, 200, 2)])
def test_chained_applications(n, k, r):
    from paper_1905_10587_gb300.api import KRR
    X, V0 = _data(n, 4, r)
    out = []
    for wait in (True, False):
        ctx = KRR(precision=1)
        ctx.build(X, 1.5, 1e-1, k, seed=3)
        V = V0.clone()
        for _ in range(8):
            V = ctx.apply_precond(V)
            if wait:
                torch.cuda.synchronize()
        out.append(V.cpu())
    assert torch.equal(out[0], out[1])
    assert torch.isfinite(out[0]).all()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,r", [(1, 1), (127, 1), (129, 1), (1025, 1), (300, 3)])
def test_solve_with_the_step_from_the_reduction(n, r, precision):
    """One column takes p . q and its step from the product's reduction, a block of columns does not.
    Bar: the tolerance, with 1e-3 of it for the float-float residual that the solve stops on."""
    from paper_1905_10587_gb300.api import KRR
    X, Y = _data(n, 4, r)
    ctx = KRR(precision=precision)
    ctx.build(X, 2.0, 1e-2, max(1, n // 10), seed=5)
    alpha, _ = ctx.solve(Y, tol=1e-6)
    Xd, a = X.double(), alpha.double().reshape(n, r)
    A = torch.exp(-torch.cdist(Xd, Xd, compute_mode="donot_use_mm_for_euclid_dist") ** 2 / 8.0)
    res = Y.double() - A @ a - 1e-2 * a
    assert (res.norm(dim=0) / Y.double().norm(dim=0)).max().item() <= 1.001e-6
