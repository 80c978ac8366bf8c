"""The first call of a process that launches a kernel also loads it.  That may
be a call captured by the caller: residual, its transpose and the stages of a step,
each captured before anything else has launched its kernels, replay to the bits
of a later eager call.  (Not capturable, first or later: cpr_step, which replays
graphs of its own; not as a first call: cpr_step_vjp, which allocates.)"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys
import torch
from paper_1709_01619_gb300 import _native as nat

dtype, eqn = int(sys.argv[1]), int(sys.argv[2])
s = torch.cuda.Stream()
with torch.cuda.stream(s):
    c = nat.Config(eqn=eqn, nx=40, ny=33, p=3, x1=8.0, y1=6.6, ax=0.8, ay=-0.5, dtype=dtype)
    q = 0.02 * torch.rand(c.shape, device="cuda", dtype=c.torch_dtype)
    if eqn == nat.EULER:
        q[0] += 1.0
        q[3] += 2.5
    w = torch.rand_like(q)
    b = [torch.zeros_like(q) for _ in range(5)]
    calls = [lambda x: x.residual(q, b[0]), lambda x: x.residual_vjp(q, w, b[1]),
             lambda x: x.step_stages(q, b[2], b[3], b[4], 0.01)]
    with nat.Context(c, stream=s) as ctx:
        s.synchronize()
        for call in calls:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                call(ctx)
            g.replay()
        s.synchronize()
        first = [x.clone() for x in b]
        for x in b:
            x.zero_()
        for call in calls:
            call(ctx)
        s.synchronize()
        assert all(torch.equal(x, y) and x.abs().sum() > 0 for x, y in zip(first, b))
print("captured first: same bits")
"""


@pytest.mark.parametrize("eqn", [0, 1])
@pytest.mark.parametrize("dtype", [0, 1])
def test_first_calls_under_capture(dtype, eqn):
    r = subprocess.run([sys.executable, "-c", CHILD, str(dtype), str(eqn)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "same bits" in r.stdout, r.stderr[-2000:]
