"""The solver's host wait for the scalars of an iteration, which the GPU writes to pinned memory."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Primary context with blocking waits; a solve of a few hundred iterations of about a millisecond each.
BLOCKING = """
import ctypes as C, sys, time
cu = C.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
assert cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0          # CU_CTX_SCHED_BLOCKING_SYNC
import torch, synth
from paper_1905_10587_gb300.api import KRR
p = synth.mixture(n=60000, k=100)
X, Y = torch.from_numpy(p.X).cuda(), torch.from_numpy(p.Y).cuda()
flags, active = C.c_uint(), C.c_int()
assert cu.cuDevicePrimaryCtxGetState(0, C.byref(flags), C.byref(active)) == 0
assert active.value and flags.value & 7 == 4, flags.value
for kw in KINDS:
    ctx = KRR(**kw)
    ctx.build(X, p.sigma, p.beta, p.k, seed=1)
    ctx.solve(Y, tol=1e-2)
    torch.cuda.synchronize()
    w, c = time.perf_counter(), time.process_time()
    _, info = ctx.solve(Y, tol=1e-5)
    torch.cuda.synchronize()
    print(time.process_time() - c, time.perf_counter() - w, info["iters"], max(info["rel_residual"]), flush=True)
"""


def test_waits_block_where_the_context_blocks():
    """Bar: half of the solve's wall time on a core; a wait that spins takes all of it, and the launches of
    an iteration about a tenth of its millisecond."""
    kinds = [dict(precision=0), dict(precision=0, recurrence=1)]
    env = dict(os.environ, PYTHONPATH=ROOT)
    res = subprocess.run([sys.executable, "-c", BLOCKING.replace("KINDS", repr(kinds))], capture_output=True, text=True,
                         env=env, cwd=ROOT, timeout=300)
    assert res.returncode == 0, res.stderr[-2000:]
    lines = [[float(v) for v in ln.split()] for ln in res.stdout.splitlines()]
    assert len(lines) == len(kinds)
    for cpu, wall, iters, rel in lines:
        assert iters > 50 and wall > 0.05 and rel <= 1e-5
        assert cpu <= 0.5 * wall, lines
