"""One-column tensor-core products that the square form does not take: two point sets, with v folded into
the exponent and as FP32 FMAs, their bounded waits, and solves that read the scalars now and then."""
import numpy as np
import pytest
import torch

from oracle import krr_oracle as O

pytestmark = pytest.mark.gpu


def _case(nr, nc, d, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    Xr, Xc = (rng.uniform(-1, 1, size=(n, d)).astype(np.float32) for n in (nr, nc))
    return Xr, Xc, rng.normal(size=nc).astype(np.float32)


# ragged sizes around the 128-row and 256-column tiles; scales at which products of v and the kernel stay
# normal.  Bars: test_gpu_parity.py's 1e-5 of the column, and 3e-5 of sum_j K_ij |v_j| for an entry.
@pytest.mark.parametrize("tc_vfold", [0, 1])
@pytest.mark.parametrize("nr,nc,d", [(1, 300, 3), (127, 257, 8), (129, 1000, 9), (700, 255, 12), (1025, 2049, 16)])
@pytest.mark.parametrize("scale", [1e-30, 1.0, 1e30])
def test_product_of_two_sets(nr, nc, d, scale, tc_vfold):
    from paper_1905_10587_gb300.api import KRR
    Xr, Xc, v = _case(nr, nc, d, nr + nc)
    v = (v * np.float32(scale)).astype(np.float32)
    v[::7] = 0.0
    q = KRR(precision=1, tc_vfold=tc_vfold).kmvm(*(torch.from_numpy(a).cuda() for a in (Xr, Xc, v)), 0.9, 0.0)
    q = q.cpu().numpy().astype(np.float64)
    Xrd, Xcd = Xr.astype(np.float64), Xc.astype(np.float64)
    K = np.exp(-((Xrd[:, None, :] - Xcd[None, :, :]) ** 2).sum(-1) / (2 * 0.9**2))
    ref, size = K @ v.astype(np.float64), K @ np.abs(v.astype(np.float64))
    assert (np.abs(q - ref) <= 3e-5 * size).all()
    if nr >= 64:
        assert np.linalg.norm(q - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("tc_vfold", [0, 1])
def test_stalled_product_of_two_sets_times_out(tc_vfold):
    from paper_1905_10587_gb300 import _lib
    from paper_1905_10587_gb300.api import KRR, KRRError
    Xr, Xc, v = _case(3000, 2500, 6, 31)
    a = [torch.from_numpy(x).cuda() for x in (Xr, Xc, v)]
    with pytest.raises(KRRError) as ei:
        KRR(precision=1, tc_vfold=tc_vfold, wait_limit_log2=20, test_stall_copies=1).kmvm(*a, 0.7, 0.0)
    assert ei.value.code == _lib.KRR_E_TIMEOUT
    torch.cuda.synchronize()
    q = KRR(precision=1, tc_vfold=tc_vfold).kmvm(*a, 0.7, 0.0).cpu().numpy()
    Xrd, Xcd = Xr.astype(np.float64), Xc.astype(np.float64)
    D = (Xrd**2).sum(1)[:, None] + (Xcd**2).sum(1)[None, :] - 2 * Xrd @ Xcd.T
    ref = np.exp(-D / (2 * 0.7**2)) @ v.astype(np.float64)
    assert np.linalg.norm(q - ref) <= 1e-5 * np.linalg.norm(ref)


# the scalars are read, and the mirror written, every few iterations only; one column takes its step from
# the product's reduction, three do not.  Bar: the solve's tolerance by the oracle's FP64 product, with
# 1e-3 of it for the float-float residual that the solve stops on.
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("check_every", [1, 2, 7, 50])
def test_solve_that_reads_now_and_then(check_every, nrhs, precision):
    import synth
    from paper_1905_10587_gb300.api import KRR
    p = synth.small(n=900, k=40)
    rng = np.random.Generator(np.random.PCG64(5))
    Y = np.concatenate([p.Y.reshape(-1, 1), rng.normal(size=(p.n, 2))], axis=1)[:, :nrhs].astype(np.float32)
    ctx = KRR(precision=precision, check_every=check_every)
    X = torch.from_numpy(p.X).cuda()
    ctx.build(X, p.sigma, p.beta, p.k, seed=1)
    for _ in range(2):                         # the second solve's first read follows the first one's last
        alpha, info = ctx.solve(torch.from_numpy(Y).cuda(), tol=1e-6)
        res = O.residual(p.X, alpha.cpu().numpy(), Y, p.sigma, p.beta)
        assert (np.linalg.norm(res, axis=0) <= 1.001e-6 * np.linalg.norm(Y, axis=0)).all()
        assert info["product_form"] == precision
