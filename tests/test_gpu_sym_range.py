"""The products of one point set with v at the ends of the FP32 range.

An infinite entry gives infinities wherever its kernel value is not zero, a sum beyond the range
gives an infinity, and one that only passes beyond it (large entries of both signs) its value."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _setup(n, d, precision):
    from paper_1905_10587_gb300.api import KRR
    g = torch.Generator(device="cuda")
    g.manual_seed(n + d)
    X = torch.rand((n, d), generator=g, device="cuda")
    v = torch.randn(n, generator=g, device="cuda")
    K = torch.exp(-torch.cdist(X.double(), X.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2 / 0.5)
    return KRR(precision=precision), X, v, K


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("n,d", [(5, 3), (256, 4), (1500, 4), (3001, 12)])
def test_infinite_entry(n, d, precision):
    ctx, X, v, _ = _setup(n, d, precision)
    v[n // 2] = math.inf
    assert torch.equal(ctx.kmvm(X, X, v, 0.5, 1e-2), torch.full((n,), math.inf, device="cuda"))
    v[n // 2] = -math.inf
    assert torch.equal(ctx.kmvm(X, X, v, 0.5, 1e-2), torch.full((n,), -math.inf, device="cuda"))
    v[0] = math.inf
    assert torch.isnan(ctx.kmvm(X, X, v, 0.5, 1e-2)).all()
    v[0] = math.nan
    assert torch.isnan(ctx.kmvm(X, X, v, 0.5, 1e-2)).all()


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_sum_beyond_the_range(precision):
    ctx, X, v, _ = _setup(1500, 4, precision)
    q = ctx.kmvm(X, X, v.abs() * 3e37, 0.5, 1e-2)
    assert torch.equal(q, torch.full_like(q, math.inf))


# 700 entries of 2e36 and then 800 of -2e36 (twice that for n = 3001): every sum of 128 is in range and
# the total is, but not the running sum.  Bar: 1e-5 of sum_j K_ij |v_j|, the bar of the parity tests for a product.
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,d", [(1500, 4), (3001, 4)])
def test_running_sum_beyond_the_range(n, d, precision):
    ctx, X, v, K = _setup(n, d, precision)
    v = torch.where(torch.arange(n, device="cuda") < 7 * n // 15, 2e36, -2e36).float()
    q = ctx.kmvm(X, X, v, 0.5, 1e-2).double()
    ref = K @ v.double() + 1e-2 * v.double()
    keep = ref.abs() < 3e38
    assert keep.any()
    assert ((q - ref).abs() <= 1e-5 * (K @ v.double().abs()))[keep].all()


# away from the ends the sums are untouched: relative to sum_j K_ij |v_j| as at scale 1
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("scale", [2.0**-110, 1.0, 2.0**110])
def test_scaled_entries(precision, scale):
    ctx, X, v, K = _setup(1500, 4, precision)
    a = ctx.kmvm(X, X, v * scale, 0.5, 1e-2).double() / scale
    ref = K @ v.double() + 1e-2 * v.double()
    assert ((a - ref).abs() <= 1e-5 * (K @ v.double().abs())).all()
