"""FP32 Euler steps (the stage updates on quads of variables, both forms of the
Runge-Kutta stages) against the FP64 oracle: every order, divergence and flux,
walls, grids below a tile, equal to one and ragged, grids of more than two CTAs
per SM, states larger than L2, and batches of such grids.

The increment of the steps is compared, so that an error of the residual shows
at its own size.  Tolerance, relative L2 of the increment d = q - q0: 1e-5 (the
FP32 residual's, on the same rough states) plus the rounding of the state, at
most 2^-24 of q for the stored result of the compensated form, and for the
Shu-Osher form for each of the three stage states of each step."""
import numpy as np
import pytest
import torch

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_parity import host, make, rough_state, to_dev

pytestmark = pytest.mark.gpu

STEPS = 2
SIZES = [(1, 1), (3, 2), (8, 8), (9, 5), (21, 19)]
MANY = (145, 133)  # more than two 8 x 8 tiles (four 8 x 4 ones) per SM
BC = [(0, 0), (1, 0), (0, 1), (1, 1)]
SCHEMES = [(div, flux) for div in (nat.DIV_LP, nat.DIV_CHAIN) for flux in (nat.RUSANOV, nat.ROE)]


def problem(p, size, bc, **kw):
    c, o = make(nat.F32, eqn=nat.EULER, nx=size[0], ny=size[1], p=p, x1=0.5 * size[0], y1=0.4 * size[1],
                bc_x=bc[0], bc_y=bc[1], **kw)
    return c, o, rough_state(o, 3, noise=0.05).astype(np.float32).astype(np.float64)


def check(got, want, q0, roundings):
    got, want, q0 = (np.asarray(x, np.float64).ravel() for x in (got, want, q0))
    d = np.linalg.norm(want - q0)
    tol = 1e-5 + roundings * 2.0 ** -24 * np.linalg.norm(want) / d
    assert np.linalg.norm(got - want) <= tol * d


DT = 0.005  # an increment of some percent of the state


@pytest.mark.parametrize("div,flux", SCHEMES)
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_steps(p, div, flux):
    """Compensated increments (cpr_step) and Shu-Osher stages (cpr_step with
    the limiter on and a bound that no element reaches)."""
    for k, size in enumerate(SIZES + [MANY]):
        c, o, q = problem(p, size, BC[k % 4], div=div, flux=flux, pts=k % 2)
        want, _, _ = oracle.run(o, q, STEPS, DT)
        with nat.Context(c) as ctx:
            d = to_dev(q, c)
            ctx.step(d, STEPS, DT)
            check(host(d), want, q, STEPS)
        c, _, _ = problem(p, size, BC[k % 4], div=div, flux=flux, pts=k % 2, limiter=1, tvb_M=1e9, lim_eps=1e-3)
        with nat.Context(c) as ctx:
            d = to_dev(q, c)
            ctx.step(d, STEPS, DT)
            assert ctx.norms(d)["n_marked"] == 0
            check(host(d), want, q, 3 * STEPS)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_step_stages(p):
    for k, size in enumerate(SIZES + [MANY]):
        c, o, q = problem(p, size, BC[k % 4], pts=k % 2)
        want, _, _ = oracle.run(o, q, 1, DT)
        with nat.Context(c) as ctx:
            d = to_dev(q, c)
            bufs = [torch.empty_like(d) for _ in range(3)]
            ctx.step_stages(d, *bufs, DT)
            check(host(bufs[2]), want, q, 3)


@pytest.mark.parametrize("p,size", [(1, (700, 640)), (2, (470, 420)), (3, (350, 315)), (4, (290, 245))])
def test_states_larger_than_l2(p, size):
    """The third stage of states whose five arrays exceed L2 takes a kernel of
    its own (it prefetches the low part)."""
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert 5 * 4 * 4 * size[0] * size[1] * (p + 1) ** 2 > l2
    c, o, q = problem(p, size, (0, 1))
    want, _, _ = oracle.run(o, q, 1, DT)
    with nat.Context(c) as ctx:
        d = to_dev(q, c)
        ctx.step(d, 1, DT)
        check(host(d), want, q, 1)


@pytest.mark.parametrize("per_instance", [False, True])
def test_batch(per_instance):
    probs = [problem(p, size, BC[(k + p) % 4]) for p in (1, 2, 3, 4) for k, size in enumerate(SIZES)]
    with nat.Batch([c for c, _, _ in probs]) as b:
        b.set_form(per_instance)
        qs = [to_dev(q, c) for c, _, q in probs]
        b.step(qs, STEPS, DT)
        for (c, o, q), d in zip(probs, qs):
            want, _, _ = oracle.run(o, q, STEPS, DT)
            check(host(d), want, q, STEPS)
