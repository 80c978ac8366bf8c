"""The FV stage kernel over the heights of its strips, which follow from the
grid, the type and the number of SMs (fv_rows in cpr_fv.cuh; 152 SMs: FP64
100 x 99 one row, 193 x 190 two, 300 x 301 four, 1001 x 999 twenty-four; FP32
below 450^2 two rows, 1001 x 999 ten, 2001 x 1701 more than thirty),
against the FP64 oracle: residual, and two fixed steps.

Tolerances: those of the other FV comparisons (FP64 1e-12, FP32 residual 1e-5,
steps 1e-6)."""
import pytest
import torch

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_fv import ORDERS, TOL32, TOL64, dev, host, make, rel, state

pytestmark = pytest.mark.gpu

CASES = [(eqn, flux, size) for eqn, flux in ((nat.EULER, nat.RUSANOV), (nat.EULER, nat.ROE), (nat.ADVECTION, nat.UPWIND))
         for size in ((1, 3), (27, 2), (100, 99), (193, 190), (300, 301))]
CASES += [(nat.EULER, nat.RUSANOV, (1001, 999)), (nat.ADVECTION, nat.RUSANOV, (1001, 999)),
          (nat.EULER, nat.RUSANOV, (2001, 1701))]


@pytest.mark.parametrize("eqn,flux,size", CASES, ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
@pytest.mark.parametrize("scheme", ORDERS)
def test_strip_heights(eqn, flux, size, dtype, scheme):
    c, o = make(dtype, scheme=scheme, eqn=eqn, flux=flux, nx=size[0], ny=size[1], x1=10.0, y1=10.0, ax=0.7, ay=-1.2,
                bc_y=nat.TRANSMISSIVE)
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


@pytest.mark.parametrize("eqn", [nat.EULER, nat.ADVECTION])
@pytest.mark.parametrize("dtype", [nat.F64, nat.F32])
@pytest.mark.parametrize("size", [(100, 99), (30, 700)])
def test_steps_after_the_end_change_nothing(eqn, dtype, size):
    """A run ends in its fourth step, shortened; the launches of further steps
    leave the state, in whichever buffer it is."""
    c, o = make(dtype, eqn=eqn, nx=size[0], ny=size[1], x1=10.0, y1=10.0, ax=0.7, ay=-1.2)
    q = state(o, "vortex", 3)
    runs = []
    for steps in (4, 5, 40):
        with nat.Context(c) as ctx:
            d = dev(q, c)
            ctx.step(d, steps, 1e-3, 3.5e-3)
            assert ctx.get_time() == (3.5e-3, 4)
            runs.append(d)
    assert torch.equal(runs[0], runs[1]) and torch.equal(runs[0], runs[2])
