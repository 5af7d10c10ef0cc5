"""The products of one point set and one column whose partial sums exceed what a context holds: several
panels.  Sampled rows against FP64, and the memory that a context takes."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _data(n, d):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    X = torch.randn((n, d), generator=g, device="cuda")
    return X, torch.randn(n, generator=g, device="cuda"), torch.randint(0, n, (200,), generator=g, device="cuda")


def _rows(X, rows, sigma):
    Xd = X.double()
    D = torch.cdist(Xd[rows], Xd, compute_mode="donot_use_mm_for_euclid_dist")
    return torch.exp(-D ** 2 / (2 * sigma * sigma))


# just past one panel and several of them; 64- and 128-wide tensor-core features
@pytest.mark.parametrize("precision,n,d", [(1, 262145, 8), (1, 700001, 4), (1, 190001, 12), (1, 400009, 10),
                                           (0, 131073, 4), (0, 300001, 8), (2, 131500, 12), (2, 270001, 3)])
def test_products_of_several_panels(precision, n, d):
    """Bars: those of the parity tests, 1e-5 of the sampled rows' norm, and 1e-5 of sum_j K_ij |v_j| for each."""
    from paper_1905_10587_gb300.api import KRR
    X, v, rows = _data(n, d)
    rows[0], rows[1] = 0, n - 1
    sigma = math.sqrt(d)
    ctx = KRR(precision=precision)
    q = ctx.kmvm(X, X, v, sigma, 1e-2)
    again = ctx.kmvm(X, X, v, sigma, 1e-2)
    assert torch.equal(q, again)
    K = _rows(X, rows, sigma)
    ref = K @ v.double() + 1e-2 * v.double()[rows]
    err = q.double()[rows] - ref
    assert err.norm() <= 1e-5 * ref.norm()
    assert (err.abs() <= 1e-5 * (K @ v.double().abs())).all()


@pytest.mark.parametrize("n,d", [(131073, 3), (200001, 8)])
def test_residual_of_several_panels(n, d):
    """Bar: 1e-11 of sum_j K_ij |a_j| (kernel values to a few 1e-12, as residual_ff.cu states)."""
    from paper_1905_10587_gb300.api import KRR
    X, y, rows = _data(n, d)
    rows[0], rows[1] = 0, n - 1
    a = torch.randn(n, device="cuda", dtype=torch.float64)
    r = KRR().residual_hp(X, y, a, math.sqrt(d), 1e-2, mode="ff")
    K = _rows(X, rows, math.sqrt(d))
    ref = y.double()[rows] - K @ a - 1e-2 * a[rows]
    assert ((r[rows] - ref).abs() <= 1e-11 * (K @ a.abs() + y.double()[rows].abs())).all()


def test_infinite_entry_and_a_solve_of_several_panels():
    from paper_1905_10587_gb300.api import KRR
    n, d = 140001, 4
    X, v, rows = _data(n, d)
    for i in (3, n - 5):                       # in the first panel and in the last
        w = v.clone()
        w[i] = math.inf
        q = KRR().kmvm(X, X, w, 2.0, 1e-2)
        assert torch.equal(q, torch.full_like(q, math.inf))
    # the step length is formed in the last panel's reduction: the solve meets its tolerance, with 1e-3
    # of it for the float-float residual that it stops on
    ctx = KRR()
    ctx.build(X, 2.0, 1.0, 300, seed=1)
    y = torch.sin(X.sum(dim=1))
    alpha, info = ctx.solve(y, tol=1e-6)
    r = ctx.residual_hp(X, y, alpha, 2.0, 1.0, mode="fp64")
    assert info["product_form"] == 0
    assert (r.norm() / y.double().norm()).item() <= 1.001e-6


@pytest.mark.parametrize("precision,n,d", [(1, 600000, 12), (0, 500000, 4)])
def test_memory_does_not_grow_with_the_square(precision, n, d):
    """Points, features and vectors are below 1 KB a point, and the partial sums below 256 MB with 8 bytes
    a point and run-times-row block beside them; without a limit these sums took 2.8 and 3.9 GB."""
    from paper_1905_10587_gb300.api import KRR
    X, v, _ = _data(n, d)
    warm = KRR(precision=precision)
    warm.kmvm(X[:100], X[:100], v[:100].contiguous(), 2.0, 0.0)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    ctx = KRR(precision=precision)
    out = torch.empty(n, device="cuda")        # the result's own memory
    before = torch.cuda.mem_get_info()[0] + out.numel() * 4
    q = ctx.kmvm(X, X, v, 2.0, 0.0)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    del q
    assert held <= n * 1024 + 300 * 2**20, held / 2**20
