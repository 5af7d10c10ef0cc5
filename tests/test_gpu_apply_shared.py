"""The preconditioner apply at anchor counts where v, held in shared memory by the pass r - F v, is
near a limit of a launch.

Every point is an anchor, so the apply is (K + beta I)^{-1}, and its backward error against K in
FP64 has the bound of test_gpu_dense.py, eta = (2 (k + 5) + k + 2) u of (||K|| + beta) ||z||."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def backward(k, nrhs, sigma=1.0, beta=1e-2):
    """Backward error over its bound, largest over the columns."""
    from paper_1905_10587_gb300.api import KRR
    g = torch.Generator(device="cuda")
    g.manual_seed(k + nrhs)
    X = torch.randn((k, 8), generator=g, device="cuda")
    V = torch.randn((k, nrhs), generator=g, device="cuda")
    ctx = KRR(pivot_tol=0.0)
    ctx.build(X, sigma, beta, k, anchors=torch.arange(k, device="cuda", dtype=torch.int32))
    z = ctx.apply_precond(V).double()
    ctx.close()
    Xd = X.double()
    K = torch.exp(-torch.cdist(Xd, Xd, compute_mode="donot_use_mm_for_euclid_dist") ** 2 / (2 * sigma**2))
    v = torch.ones(k, dtype=torch.float64, device="cuda")
    for _ in range(30):                       # a lower bound of ||K||: the test is no easier for it
        v = K @ (v / v.norm())
    r = (K @ z + beta * z - V.double()).norm(dim=0)
    eta = (2 * (k + 5) + k + 2) * 2.0**-24
    return (r / (eta * (v.norm() + beta) * z.norm(dim=0))).max().item()


# sizes at which the pass needs just under 48 KB beside its static shared memory, each in a process
# that has not run a larger one before
NEAR_48K = [(1504, 8), (1536, 8), (1736, 7), (2048, 6), (2432, 5), (3060, 4)]


def test_apply_just_below_48_kilobytes():
    code = "import test_gpu_apply_shared as t\nfor k, r in t.NEAR_48K:\n    print(k, r, t.backward(k, r), flush=True)\n"
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, cwd=ROOT, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
    got = [line.split() for line in res.stdout.splitlines()]
    assert len(got) == len(NEAR_48K)
    for k, r, e in got:
        assert float(e) <= 1.0, (k, r, e)


# from about 7200 anchors eight columns do not fit the shared memory of a block; 7 + 2 columns at k = 8000
@pytest.mark.parametrize("k,nrhs", [(7100, 8), (8000, 8), (8000, 9)])
def test_apply_with_many_anchors(k, nrhs):
    assert backward(k, nrhs) <= 1.0


# partial sums of F^T r from every number of blocks up to the most there are (four an SM), with few and
# many columns a pass; the backward error against the Nystrom K~ of the same anchors in FP64
@pytest.mark.parametrize("nrhs", [1, 2, 3, 8])
@pytest.mark.parametrize("n,k", [(33, 20), (1025, 90), (20011, 600), (60013, 300)])
def test_apply_partial_sums(n, k, nrhs, sigma=1.0, beta=1e-2):
    from paper_1905_10587_gb300.api import KRR
    g = torch.Generator(device="cuda")
    g.manual_seed(n + nrhs)
    X = torch.randn((n, 8), generator=g, device="cuda")
    V = torch.randn((n, nrhs), generator=g, device="cuda")
    ctx = KRR(pivot_tol=0.0)
    ctx.build(X, sigma, beta, k, anchors=torch.arange(k, device="cuda", dtype=torch.int32))
    z = ctx.apply_precond(V).double()
    ctx.close()
    Xd = X.double()
    C = torch.exp(-torch.cdist(Xd, Xd[:k], compute_mode="donot_use_mm_for_euclid_dist") ** 2 / (2 * sigma**2))
    L = torch.linalg.cholesky(C[:k])
    F = torch.linalg.solve_triangular(L, C.t(), upper=False)
    v = torch.ones(n, dtype=torch.float64, device="cuda")
    for _ in range(30):                       # a lower bound of ||K~||
        v = F.t() @ (F @ (v / v.norm()))
    r = (F.t() @ (F @ z) + beta * z - V.double()).norm(dim=0)
    eta = (2 * (k + 5) + k + 2) * 2.0**-24
    assert (r / (eta * (v.norm() + beta) * z.norm(dim=0))).max().item() <= 1.0
