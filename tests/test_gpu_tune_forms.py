"""Tuned entries of one column: the product of one point set and the product of two are different
kernels, and neither takes the other's entry."""
import math
import time

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _built(api, precision, **opts):
    p = synth.mixture(n=20000, k=200)
    X = torch.from_numpy(p.X).cuda()
    ctx = api.KRR(precision=precision, **opts)
    ctx.build(X, p.sigma, p.beta, p.k, seed=1)
    return p, X, ctx


def _key(form, width, n):
    return f"form={form} w={width} r=1 lg={int(math.floor(math.log2(n)))}"


def _ms(f):
    f()
    best = math.inf
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(5):
            f()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_one_column_autotune_leaves_two_set_products_fast(precision):
    """A product of two sets of the tuned size takes column splits that were timed for it: not slower
    than the cost model's by more than timing noise (bar: half as long again)."""
    from paper_1905_10587_gb300 import api
    api.tune_clear()
    p, X, ctx = _built(api, precision)
    splits, _, _ = ctx.autotune(nrhs=1, reps=2)
    width = 64 if precision == 1 else 8
    assert api.tune_get(_key(precision, width, p.n))[0] == splits
    height = api.tune_get(_key(3, width, p.n))
    assert (height is not None) == (precision == 1)
    if height:
        assert 1 <= height[0] <= 4 and height[1] == 0
    Z = X.clone()                              # the same points, but another set
    v = torch.randn(p.n, device="cuda")
    plain, tuned = api.KRR(precision=precision), api.KRR(precision=precision, autotune=1)
    a = _ms(lambda: plain.kmvm(Z, X, v, p.sigma, 0.0))
    b = _ms(lambda: tuned.kmvm(Z, X, v, p.sigma, 0.0))
    api.tune_clear()
    assert b <= 1.5 * a, (splits, a, b)


@pytest.mark.parametrize("entry", [(12, 0), (64, 0), (6, 1)])
def test_entries_of_two_set_products_leave_the_square_one_alone(entry):
    """An entry of the form for two sets (a table of an earlier version holds them) changes no bit of the
    product of one set; its own entry only cuts the work differently."""
    from paper_1905_10587_gb300 import api
    p, X, ctx = _built(api, 1)
    v = torch.randn(p.n, device="cuda")
    tuned = api.KRR(precision=1, autotune=1)
    api.tune_clear()
    q = ctx.kmvm(X, X, v, p.sigma, p.beta)
    assert torch.equal(tuned.kmvm(X, X, v, p.sigma, p.beta), q)
    api.tune_set(_key(1, 64, p.n), entry[0], entry[1], 1.0)
    assert torch.equal(tuned.kmvm(X, X, v, p.sigma, p.beta), q)
    api.tune_set(_key(3, 64, p.n), entry[0], entry[1], 1.0)
    r = tuned.kmvm(X, X, v, p.sigma, p.beta)
    api.tune_clear()
    # both are within 1e-5 of the product (test_gpu_parity.py)
    assert ((r - q).norm() / q.norm()).item() <= 2e-5
