"""The pivoted QR at row lengths around its kernels' widths (a lane's 2, 4, 8, ... values of a row,
one and several values of a reflector's thread, rows of a warp that are missing), and with squares
outside the range of the float-float pairs, which are summed in FP64 instead.

Bar: that of test_gpu_parity.py's pivot tests: every choice maximal by the FP64 replay up to 1e-5 of
the largest norm (FP32 residuals, at most 40 reflectors of 2^-24 each with a margin), R_jj too."""
import numpy as np
import pytest
import torch

from oracle import krr_oracle as O

pytestmark = pytest.mark.gpu


def _check(n, l, k, scale):
    from paper_1905_10587_gb300.api import KRR
    rng = np.random.Generator(np.random.PCG64(n + l))
    Y = (rng.normal(size=(n, l)) * np.logspace(0, -2, l) * scale).astype(np.float32)
    if n > 9:
        Y[9] = 0.0   # a row without a norm
    piv, rd = KRR().qrcp(torch.from_numpy(Y).cuda(), k)
    piv, rd = piv.cpu().numpy(), rd.cpu().numpy().astype(np.float64)
    got, best = O.qrcp_replay(Y.T.astype(np.float64), piv)
    tol = 1e-5 * best[0]
    assert len(set(piv.tolist())) == k
    assert np.all(got >= best - tol)
    np.testing.assert_allclose(rd, got, rtol=0, atol=tol)


@pytest.mark.parametrize("n,l,k", [(1, 1, 1), (7, 3, 3), (8, 8, 8), (65, 31, 31), (1023, 33, 33), (301, 64, 40),
                                   (130, 129, 34), (257, 257, 33), (200, 513, 33), (77, 1024, 34), (90, 1056, 40),
                                   (70, 2049, 35), (40, 4096, 20)])
def test_row_lengths(n, l, k):
    _check(n, l, k, 1.0)


@pytest.mark.parametrize("scale", [2.0**-50, 2.0**60])
@pytest.mark.parametrize("n,l,k", [(500, 40, 36), (70, 1040, 36)])
def test_squares_outside_float_range(n, l, k, scale):
    _check(n, l, k, scale)
