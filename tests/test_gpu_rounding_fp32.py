"""Rounding of the FP32 steps.

Shu-Osher stages of a vanishing step leave the state's bits alone.

Advection: the error of a run against the FP64
oracle is at most that of the same scheme written plainly in FP32 (flux
derivative by the rows of D, edge values of the flux, corrections, the stages
as compensated increments, each table entry and factor rounded once), on the
same states.

An operator entry or a factor rounded once more is an error common to every
element and step: it does not average out, and shows as a speed of the wave.

Tolerance: 1.25 times the plain form's error, both as root mean square over
eight states; the square of one state's error is a sum over the rounding of
a few entries and factors, common to all states, and of many independent ones
(thousands of values), so the ratio has no spread of that size."""
import numpy as np
import pytest
import torch

import oracle
from paper_1709_01619_gb300 import _native as nat
from test_gpu_parity import host, make, rough_state, to_dev

pytestmark = pytest.mark.gpu

F = np.float32


def tables(n):
    """D, l(-1), l(+1), g_L', g_R' on Gauss points, rounded to FP32."""
    x = np.polynomial.legendre.leggauss(n)[0]
    P = np.polynomial.polynomial.Polynomial
    basis = [np.prod([P([-x[m], 1.0]) / (x[l] - x[m]) for m in range(n) if m != l] or [P([1.0])]) for l in range(n)]
    leg = np.polynomial.legendre.Legendre.basis
    g = ((-1.0) ** n * 0.5 * (leg(n) - leg(n - 1))).deriv()
    return (np.array([[b.deriv()(a) for b in basis] for a in x]).astype(F), np.array([b(-1.0) for b in basis]).astype(F),
            np.array([b(1.0) for b in basis]).astype(F), g(x).astype(F), (-g(-x)).astype(F))


def plain_residual(c, tab, q):
    """-(div f) of q[j, i, b, a], periodic, both velocities positive, upwind."""
    D, lm, lp, dgl, dgr = tab

    def line(q, a, axis):  # the line's points on the last axis
        f = F(a) * q
        fL, fR, up = f @ lm, f @ lp, F(a) * (q @ lp)
        low = np.roll(up, 1, axis)
        return f @ D.T + (low - fL)[..., None] * dgl + (up - fR)[..., None] * dgr

    rx, ry = line(q, c.ax, 1), line(q.swapaxes(2, 3), c.ay, 0).swapaxes(2, 3)
    return -F(2.0 * c.nx / (c.x1 - c.x0)) * rx - F(2.0 * c.ny / (c.y1 - c.y0)) * ry


def plain_run(c, q, steps, dt):
    tab, dt = tables(c.p + 1), F(dt)
    hi = q.astype(F).reshape(c.ny, c.nx, c.p + 1, c.p + 1)
    lo = np.zeros_like(hi)
    for _ in range(steps):
        b1 = dt * plain_residual(c, tab, hi)
        b2 = F(0.25) * (b1 + dt * plain_residual(c, tab, hi + b1))
        d = F(2.0 / 3.0) * (b2 + dt * plain_residual(c, tab, hi + b2))
        s = hi + d  # two-sum, then the low parts folded back
        t = s - hi
        e = ((hi - (s - t)) + (d - t)) + lo
        hi = s + e
        lo = e - (hi - s)
    return hi.astype(np.float64).reshape(q.shape)


@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_advection_error_at_most_the_plain_form(p):
    c, o = make(nat.F32, eqn=nat.ADVECTION, nx=48, ny=45, p=p, ax=1.0, ay=1.0, flux=nat.UPWIND)
    x, y = oracle.point_coords(o)
    dt, steps = {1: 0.15, 2: 0.1, 3: 0.06, 4: 0.04}[p] / 48 / np.sqrt(2.0), 100
    rng = np.random.default_rng(p)
    got, plain = [], []
    with nat.Context(c) as ctx:
        for _ in range(8):
            sx, sy = rng.uniform(0.0, 1.0, 2)
            q = rng.uniform(0.5, 1.5) * np.sin(2 * np.pi * (x + sx)) * np.sin(2 * np.pi * (y + sy))
            q = q[None].astype(F).astype(np.float64)
            want, _, _ = oracle.run(o, q, steps, dt)
            d = to_dev(q, c)
            ctx.step(d, steps, dt)
            norm = np.linalg.norm(want)
            got.append(np.linalg.norm(host(d).reshape(want.shape) - want) / norm)
            plain.append(np.linalg.norm(plain_run(c, q, steps, dt) - want) / norm)
    rms = [float(np.sqrt(np.mean(np.square(v)))) for v in (got, plain)]
    assert rms[0] <= 1.25 * rms[1], rms


@pytest.mark.parametrize("eqn", [nat.EULER, nat.ADVECTION])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_stage_weights_sum_to_one(p, eqn):
    """60 steps of size 1e-30 (every increment is far below the last place of
    the state) with the limiter on (which marks nothing): the Shu-Osher stages
    only average a state with itself, so its bits stay."""
    c, o = make(nat.F32, eqn=eqn, nx=21, ny=13, p=p, x1=10.0, y1=6.0, limiter=1, tvb_M=1e9, lim_eps=1e-3, ax=0.7, ay=-0.4)
    q = to_dev(rough_state(o, 3, noise=0.05), c)
    with nat.Context(c) as ctx:
        d = q.clone()
        ctx.step(d, 60, 1e-30)
    assert torch.equal(d, q)
