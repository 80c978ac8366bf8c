"""The tiles of the FP64 Euler, advection and adjoint kernels at their edges:
grids smaller than a tile, equal to one, one element more, and large enough
for the FP64 rule to pick each of its tiles (4 x 2 for p = 4, 4 x 4, 8 x 4),
with both kinds of boundary, against the FP64 oracle.

Tolerances (those of the other comparisons): FP64 1e-12 relative L2 (rounding
order only); FP32 residual 1e-5, fixed steps 1e-6."""
import numpy as np
import pytest

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_parity import TOL32, TOL64, host, make, rel_l2, rough_state, to_dev

pytestmark = pytest.mark.gpu

SMALL = [(1, 1), (3, 2), (4, 4), (5, 3), (8, 4), (9, 5)]
LARGE = {1: (131, 133), 2: (131, 133), 3: (97, 99), 4: (75, 77)}
BC = [(0, 0), (1, 0), (0, 1), (1, 1)]


def check(dtype, p, size, bc, steps=2, **kw):
    c, o = make(dtype, nx=size[0], ny=size[1], p=p, x1=6.0, y1=5.0, bc_x=bc[0], bc_y=bc[1], **kw)
    q = rough_state(o, 7)
    if dtype == nat.F32:
        q = q.astype(np.float32).astype(np.float64)
    r = oracle.residual(o, q)
    qn, _, _ = oracle.run(o, q, steps, 1e-4)
    with nat.Context(c) as ctx:
        d = to_dev(q, c)
        assert rel_l2(host(ctx.residual(d)), r) <= (TOL64 if dtype == nat.F64 else TOL32)
        ctx.step(d, steps, 1e-4)
        assert rel_l2(host(d), qn) <= (TOL64 if dtype == nat.F64 else 1e-6)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("div", [nat.DIV_LP, nat.DIV_CHAIN])
@pytest.mark.parametrize("flux", [nat.RUSANOV, nat.ROE])
def test_euler_fp64(p, div, flux):
    for k, size in enumerate(SMALL + [(21, 19), (48, 40)]):
        check(nat.F64, p, size, BC[k % 4], eqn=nat.EULER, pts=k % 2, div=div, flux=flux)
    check(nat.F64, p, LARGE[p], (0, 1), eqn=nat.EULER, div=div, flux=flux)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
@pytest.mark.parametrize("velocity", [(0.7, 1.3), (-0.7, 0.4), (0.6, -1.1), (-0.3, -0.9), (0.0, 0.5)])
def test_advection(p, dtype, velocity):
    for k, size in enumerate(SMALL + [(21, 19), LARGE[p]]):
        check(dtype, p, size, BC[k % 4], eqn=nat.ADVECTION, pts=k % 2, div=k // 2 % 2,
              flux=(nat.UPWIND, nat.RUSANOV)[k % 2], ax=velocity[0], ay=velocity[1])


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
def test_euler_adjoint(p, dtype):
    for k, size in enumerate(SMALL + [(21, 18)]):
        bc = BC[k % 4]
        c, o = make(dtype, eqn=nat.EULER, nx=size[0], ny=size[1], p=p, x1=6.0, y1=5.0, bc_x=bc[0], bc_y=bc[1],
                    pts=k % 2)
        q = rough_state(o, 9)
        w = np.random.default_rng(k).standard_normal(q.shape)
        if dtype == nat.F32:
            q, w = q.astype(np.float32).astype(np.float64), w.astype(np.float32).astype(np.float64)
        with nat.Context(c) as ctx:
            got = host(ctx.residual_vjp(to_dev(q, c), to_dev(w, c)))
        assert rel_l2(got, oracle.residual_vjp(o, q, w)) <= (TOL64 if dtype == nat.F64 else TOL32)
