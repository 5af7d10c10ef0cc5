"""The symmetric products (one right-hand side, square, each pair evaluated once) against the
FP64 oracle: tile and row-block edges, every feature width, every work split, and
columns far from unit scale.

Tolerances are those of the products' other tests: 1e-5 of the column norm, and per
entry 3e-5 of sum_j |K_ij v_j| (the expansion's rounding, see test_gpu_parity.py).
"""
import numpy as np
import pytest
import torch

from oracle import krr_oracle as O

pytestmark = pytest.mark.gpu


def _case(n, d, seed=5):
    rng = np.random.Generator(np.random.PCG64(seed))
    X = rng.normal(size=(n, d)).astype(np.float32)
    v = rng.normal(size=(n, 1)).astype(np.float32)
    return X, v, 0.6 * float(np.sqrt(d)), 1e-2


def _product(X, v, sigma, beta, precision=1, **opts):
    from paper_1905_10587_gb300.api import KRR
    Xd, vd = torch.from_numpy(X).cuda(), torch.from_numpy(v).cuda()
    ctx = KRR(precision=precision, **opts)
    return ctx.kmvm(Xd, Xd, vd[:, 0], sigma, beta).cpu().numpy().astype(np.float64)


def _check(q, X, v, sigma, beta):
    ref = O.kmvm(X, v.astype(np.float64), sigma, beta)[:, 0]
    mag = O.kmvm(X, np.abs(v.astype(np.float64)), sigma, beta)[:, 0]
    assert np.linalg.norm(q - ref) <= 1e-5 * np.linalg.norm(ref)
    assert np.all(np.abs(q - ref) <= 3e-5 * mag)


# 1, 127 and 257 are single tiles and units; 2049, 2303 .. 2305 straddle tiles, units and row blocks;
# d = 1, 2, 5, 7, 9 use 1 to 4 K steps of 256-column units, d = 10, 12, 16 5 to 7 of 128-column ones
@pytest.mark.parametrize("n,d", [(1, 4), (127, 3), (257, 11), (2048, 1), (2049, 2), (2303, 5), (2304, 7), (2305, 9), (2049, 10),
                                 (2561, 12), (4100, 16), (9001, 8)])
def test_symmetric_product_matches_the_oracle(n, d):
    X, v, sigma, beta = _case(n, d)
    q = _product(X, v, sigma, beta)
    _check(q, X, v, sigma, beta)


# FP32 forms: 128-column tiles, 256-row blocks; four rows per thread for differences above d = 10,
# an odd number of staged values per column (d odd or even by form), d = 4, 8, 12, 16 with a packed
# row that ends in the norm or spills into the next float4
@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("n,d", [(1, 3), (127, 1), (128, 4), (129, 8), (255, 2), (257, 11), (1000, 7), (2305, 10),
                                 (4099, 12), (3000, 16), (9001, 3)])
def test_symmetric_fp32_products_match_the_oracle(n, d, precision):
    X, v, sigma, beta = _case(n, d)
    _check(_product(X, v, sigma, beta, precision=precision), X, v, sigma, beta)


@pytest.mark.parametrize("precision", [0, 2])
def test_fp32_results_do_not_depend_on_timing(precision):
    X, v, sigma, beta = _case(5000, 8)
    first = _product(X, v, sigma, beta, precision=precision)
    for _ in range(3):
        assert np.array_equal(first, _product(X, v, sigma, beta, precision=precision))


@pytest.mark.parametrize("d,width", [(4, 64), (11, 128)])
@pytest.mark.parametrize("split", [1, 2, 3, 4])
def test_every_row_block_height(d, width, split):
    from paper_1905_10587_gb300 import api
    n = 3333
    X, v, sigma, beta = _case(n, d)
    api.tune_clear()
    try:
        api.tune_set(f"form=1 w={width} r=1 lg=11", split)
        q = _product(X, v, sigma, beta, autotune=1)
    finally:
        api.tune_clear()
    _check(q, X, v, sigma, beta)


@pytest.mark.parametrize("scale", [0.0, 1e-38, 1e-30, 1e30])
def test_columns_far_from_unit_scale(scale):
    X, v, sigma, beta = _case(2500, 3)
    v = (v * np.float32(scale)).astype(np.float32)
    q = _product(X, v, sigma, beta)
    if scale == 0.0:
        assert not np.any(q)
    else:
        _check(q, X, v, sigma, beta)


def test_points_and_vector_at_odd_addresses():
    # a vector that starts 4 bytes past a 16-byte boundary
    from paper_1905_10587_gb300.api import KRR
    X, v, sigma, beta = _case(2100, 6)
    Xd = torch.from_numpy(X).cuda()
    buf = torch.zeros(2101, device="cuda")
    buf[1:] = torch.from_numpy(v[:, 0]).cuda()
    q = KRR(precision=1).kmvm(Xd, Xd, buf[1:], sigma, beta).cpu().numpy().astype(np.float64)
    _check(q, X, v, sigma, beta)


def test_results_do_not_depend_on_timing():
    X, v, sigma, beta = _case(5000, 8)
    first = _product(X, v, sigma, beta)
    for _ in range(3):
        again = _product(X, v, sigma, beta)
        assert np.array_equal(first, again)


# the float-float residual with one column: units of 64 x 64, 128 x 128 and 256 x 128 pairs (taken as
# n grows), their edges, and odd and even strides of the staged points; bar as in test_gpu_parity.py
@pytest.mark.parametrize("n,d", [(1, 2), (63, 1), (64, 8), (65, 16), (129, 5), (257, 4), (1000, 16), (3001, 3),
                                 (7000, 2), (13001, 1)])
def test_symmetric_residual(n, d):
    from paper_1905_10587_gb300.api import KRR
    rng = np.random.Generator(np.random.PCG64(31 * d + n))
    X = (rng.normal(size=(n, d)) * 2 + 5).astype(np.float32)
    A = rng.normal(size=(n, 1)) * 100
    Y = rng.normal(size=(n, 1)).astype(np.float32)
    sigma, beta = 0.4 * float(np.sqrt(d)), 1e-3
    R = KRR().residual_hp(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), torch.from_numpy(A).cuda(), sigma,
                          beta, mode="ff").cpu().numpy()
    rows = rng.choice(n, min(n, 1500), replace=False)
    ref = Y[rows].astype(np.float64) - O.kmvm(X, A, sigma, 0.0, rows=rows) - beta * A[rows]
    cond = O.kmvm(X, np.abs(A), sigma, 0.0, rows=rows) + beta * np.abs(A[rows]) + np.abs(Y[rows])
    assert np.all(np.abs(R[rows] - ref) <= 2e-11 * cond)
