"""FV steps around an element that holds NaN: minmod takes a NaN difference as
no slope, so in one residual only the elements that share a face with it turn
NaN, and every other one has the oracle's value.

Tolerances: those of the other FV comparisons (FP64 1e-12, FP32 1e-5)."""
import numpy as np
import pytest

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_fv import ORDERS, TOL32, TOL64, dev, host, make, rel, state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
@pytest.mark.parametrize("scheme", ORDERS)
@pytest.mark.parametrize("eqn", [nat.EULER, nat.ADVECTION])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_nan_stays_with_the_elements_that_share_a_face(dtype, scheme, eqn, sign):
    # the element in the ring of a neighbouring strip (28 columns) and inside one
    for i, j in ((28, 9), (11, 4)):
        c, o = make(dtype, scheme=scheme, eqn=eqn, nx=61, ny=19, x1=10.0, y1=3.0, ax=0.7, ay=-1.2)
        q = state(o, "vortex", 6)
        if dtype == nat.F32:
            q = q.astype(np.float32).astype(np.float64)
        q = np.asarray(q).reshape(c.shape).copy()
        q[-1, j * c.nx + i] = np.copysign(np.nan, sign)
        want = oracle.residual(o, q).reshape(c.shape[0], c.ny, c.nx)
        with nat.Context(c) as ctx:
            got = host(ctx.residual(dev(q, c))).reshape(want.shape)
        # (which variables of those turn NaN depends on how a zero times NaN is
        # written in the flux)
        near = np.zeros(want.shape[1:], dtype=bool)
        near[j, i - 1:i + 2] = near[j - 1:j + 2, i] = True
        assert not np.isnan(want[:, ~near]).any() and np.isnan(want[-1, j, i])
        assert not np.isnan(got[:, ~near]).any() and np.isnan(got[-1, j, i])
        ok = ~np.isnan(want) & ~np.isnan(got)
        assert rel(got[ok], want[ok]) <= (TOL64 if dtype == nat.F64 else TOL32)
