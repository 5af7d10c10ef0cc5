"""Centring and packing: products of points far from the origin, where a wrong mean or a wrong
packed coordinate shows as cancellation in the expansion.  Sizes around the mean kernels' block
of 256 threads and the feature tile of 128 points; dimensions that do not divide 256 and the
padded ones above 16.

Bar: 1e-5 of sum_j |K_ij v_j| per entry.  With points within 4 sigma of their mean the expansion
rounds terms of size ||x_h||^2 <= ~25 d / d, about 3e-6 relative; without centring (offset 40) they
would be 100 times that size.
"""
import numpy as np
import pytest
import torch

from oracle import krr_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 129, 256, 257, 3001])
@pytest.mark.parametrize("d,precision", [(1, 0), (3, 1), (7, 1), (12, 1), (16, 1), (5, 0), (17, 0), (33, 0), (64, 0),
                                         (11, 2)])
def test_offset_points(n, d, precision):
    from paper_1905_10587_gb300.api import KRR
    rng = np.random.Generator(np.random.PCG64(100 * d + n))
    X = (40.0 + rng.normal(size=(n, d))).astype(np.float32)
    v = rng.normal(size=(n, 1)).astype(np.float32)
    sigma = float(np.sqrt(d))
    Xd, vd = torch.from_numpy(X).cuda(), torch.from_numpy(v).cuda()
    q = KRR(precision=precision).kmvm(Xd, Xd, vd, sigma, 0.0).cpu().numpy().astype(np.float64)
    ref = O.kmvm(X, v.astype(np.float64), sigma, 0.0)
    mag = O.kmvm(X, np.abs(v).astype(np.float64), sigma, 0.0)
    assert np.all(np.abs(q - ref) <= 1e-5 * mag)
