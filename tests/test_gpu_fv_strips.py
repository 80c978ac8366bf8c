"""The FV stage kernel at the edges of its strips (28 columns of elements per
warp; 2 to 32 rows, by the size of the grid): grids one column short of, equal
to and one past a strip, ragged in both directions, and large enough for
strips of 4 and 16 rows, against the FP64 oracle.

Tolerances (those of the other FV comparisons): FP64 1e-12 relative L2
(rounding order only); FP32 residual 1e-5 and fixed steps 1e-6."""
import pytest
import torch

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_fv import ORDERS, TOL32, TOL64, dev, host, make, rel, state

pytestmark = pytest.mark.gpu

SIZES = [(27, 3), (28, 2), (29, 5), (57, 7), (3, 33), (565, 501), (1541, 801)]


@pytest.mark.parametrize("size", SIZES, ids=lambda s: f"{s[0]}x{s[1]}")
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
@pytest.mark.parametrize("scheme", ORDERS)
@pytest.mark.parametrize("wall", [False, True])
def test_strip_edges(size, dtype, scheme, wall):
    bc = nat.TRANSMISSIVE if wall else nat.PERIODIC
    c, o = make(dtype, scheme=scheme, eqn=nat.EULER, nx=size[0], ny=size[1], x1=10.0, y1=10.0, bc_x=bc, bc_y=bc)
    q = state(o, "vortex", 3)
    if dtype == nat.F32:
        q = q.astype("float32").astype("float64")
    R_or = oracle.residual(o, q)
    q_or, _, _ = oracle.run(o, q, 2, 1e-4)
    with nat.Context(c) as ctx:
        d = dev(q, c)
        assert rel(host(ctx.residual(d)), R_or) <= (TOL64 if dtype == nat.F64 else TOL32)
        ctx.step(d, 2, 1e-4)
        assert rel(host(d), q_or) <= (TOL64 if dtype == nat.F64 else 1e-6)
    torch.cuda.synchronize()
