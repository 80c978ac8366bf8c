"""The limiter's shortcut for flat elements (a warp whose elements cannot be
marked leaves out the edge test): states whose elements deviate from their
averages by amounts on both sides of the shortcut's bound, in stretches of
flat, of varied and of steep elements, with the bound set by eps, by M h^2 or
zero, against the FP64 oracle.

Marks are compared where the oracle's margin is farther from zero than the
arithmetic moves it: 64 roundings of the largest value (FP64 about 1e-14,
FP32 about 4e-6 for values below 10); the limited state as elsewhere (FP64
1e-12, FP32 1e-5)."""
import numpy as np
import pytest

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_parity import TOL32, TOL64, host, make, rel_l2, to_dev

pytestmark = pytest.mark.gpu


def state(o, seed):
    rng = np.random.default_rng(seed)
    e = np.arange(o.ne)
    amp = np.where(e % 192 < 96, 1e-6, np.where(e % 192 < 160, 10.0 ** rng.uniform(-4.5, -2.0, o.ne), 0.05))
    q = np.empty((4, o.ne, o.n * o.n))
    for v, base in enumerate((1.0, 0.3, -0.2, 2.5)):
        q[v] = base + amp[:, None] * rng.uniform(-1.0, 1.0, (o.ne, o.n * o.n))
    return q


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
@pytest.mark.parametrize("bound", [(50.0, 1e-3), (0.0, 1e-3), (0.0, 0.0), (4.0, 1e-6)])
def test_marks_on_both_sides_of_the_bound(p, dtype, bound):
    c, o = make(dtype, eqn=nat.EULER, nx=51, ny=37, p=p, x1=1.0, y1=0.7, bc_x=1, limiter=1, tvb_M=bound[0],
                lim_eps=bound[1])
    q = state(o, p)
    if dtype == nat.F32:
        q = q.astype(np.float32).astype(np.float64)
    q_or, marks_or, margin, _ = oracle.limit(o, q)
    with nat.Context(c) as ctx:
        d = to_dev(q, c)
        ctx.limit(d)
        marks, ql = ctx.get_marks(), host(d)
    u = 2.0 ** -53 if dtype == nat.F64 else 2.0 ** -24
    sure = np.abs(margin) > 64 * u * np.abs(q).max()
    assert np.array_equal(marks[sure], marks_or[sure])
    if bound[1] > 0:
        assert 0 < marks.sum() < o.ne
    agree = marks == marks_or
    assert rel_l2(ql[:, agree, :], q_or[:, agree, :]) <= (TOL64 if dtype == nat.F64 else TOL32)
