"""A build whose Cholesky refuses a pivot keeps the anchors before it: the same preconditioner, bit for
bit, as from those anchors alone, wherever in the 32-column blocks the pivot lies, and whatever the
workspace held before."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [1, 2, 31, 32, 33, 63, 64, 65, 100, 129])
def test_build_with_a_repeated_anchor(at):
    from paper_1905_10587_gb300.api import KRR
    n, k, d = 700, 160, 4
    g = torch.Generator(device="cuda")
    g.manual_seed(at)
    X = torch.randn((n, d), generator=g, device="cuda")
    V = torch.randn((n, 2), generator=g, device="cuda")
    S = torch.randperm(n, generator=g, device="cuda")[:k].to(torch.int32)
    S[at] = S[at // 2]                         # its pivot is the rounding of 1 - 1
    fresh, used, only = KRR(), KRR(), KRR()
    used.build(X, 0.3, 1e-2, k, anchors=torch.arange(k, device="cuda", dtype=torch.int32))
    out = []
    for ctx, T in ((fresh, S), (used, S), (only, S[:at].contiguous())):
        ctx.build(X, 0.3, 1e-2, T.numel(), anchors=T)
        assert torch.equal(ctx.anchors(), S[:at])
        out.append(ctx.apply_precond(V))
        assert torch.isfinite(out[-1]).all()
        ctx.close()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
