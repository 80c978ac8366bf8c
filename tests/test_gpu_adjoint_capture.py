"""The step adjoint's launches under stream capture: kernels launched behind
one another with programmatic dependence keep their order in a graph."""
import numpy as np
import pytest
import torch

from paper_1709_01619_gb300 import _native as nat
from test_gpu_adjoint import dev, make, rough

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eqn", [0, 1])
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
def test_step_adjoint_under_capture(eqn, dtype):
    """The launches of a step's stages and of its transpose, captured in a
    graph and replayed twice, give the bits of the eager calls."""
    c, o = make(dtype, eqn=eqn, nx=40, ny=33, p=3, x1=8.0, y1=6.6, ax=0.8, ay=-0.5)
    q, w = rough(o, 5), np.random.default_rng(6).standard_normal(c.shape)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        qd, wd = dev(q, c), dev(w, c)
        bufs = [torch.empty_like(qd) for _ in range(4)]
        with nat.Context(c, stream=s) as ctx:
            def call():
                ctx.step_stages(qd, *bufs[:3], 0.01)
                ctx.step_vjp_stages(qd, bufs[0], bufs[1], wd, 0.01, bufs[3])
            call()
            s.synchronize()
            ref = [b.clone() for b in bufs]
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                call()
            for _ in range(2):
                for b in bufs:
                    b.zero_()
                g.replay()
                s.synchronize()
                assert all(torch.equal(a, b) for a, b in zip(ref, bufs))
