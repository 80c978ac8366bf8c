"""The workloads that a user of this framework has it do, as measurable cases.

listed() names them, draw(rng) gives more of the same ranges, prepare(case,
seed) makes what a program has in hand before the call (the solver context or
batch and the initial state), run(state) is one pass through the public entry
points, work(case) the bytes and operations of the method, and exact(case,
seed) the same pass in plain 64-bit torch, written here from the formulas of
the scheme without the package's code.

A time-stepping pass starts from the prepared initial state (copied over the
working state, as a driver that restarts a solve does) and takes a number of
SSP-RK3 steps.
"""
import math

import numpy as np
import torch

from paper_1709_01619_gb300 import _native as nat
from paper_1709_01619_gb300 import adjoint

GAMMA = 1.4
PTS = {"gauss": nat.GAUSS, "lobatto": nat.LOBATTO}
DIV = {"lp": nat.DIV_LP, "chain": nat.DIV_CHAIN}
FLUX = {"rusanov": nat.RUSANOV, "upwind": nat.UPWIND, "roe": nat.ROE}
CORR = {"gdg": nat.CORR_GDG, "ndg": nat.CORR_NDG}
SCHEME = {"cpr": nat.SCHEME_CPR, "fv2": nat.SCHEME_FV_MUSCL, "fv3": nat.SCHEME_FV_MUSCL3}
# CFL numbers the repository's workloads use per order (FV: p = 0)
CFL = {0: 0.4, 1: 0.15, 2: 0.1, 3: 0.06, 4: 0.04}


def _case(name=None, **kw):
    c = {"kind": "step", "problem": "vortex", "scheme": "cpr", "nx": 128, "ny": 128, "p": 3, "dtype": "f32",
         "pts": "gauss", "div": "lp", "flux": "rusanov", "corr": "gdg", "limiter": False, "steps": 1, "fixed": False}
    c.update(kw)
    if name is not None:
        c = {"name": name, **c}
    return c


def listed():
    return [
        # one right-hand side for a caller with its own time integrator on a
        # small odd grid: the smallest call, latency only
        _case("residual_45x37_p2_f32", kind="residual", nx=45, ny=37, p=2, steps=0),
        # the linear advection validation run: 16^2, p = 2, one period in 227
        # equal FP64 steps (hundreds of tiny stages, launch latency)
        _case("advection_16_p2_f64_227", problem="sine", nx=16, ny=16, p=2, dtype="f64", steps=227, fixed=True),
        # the isentropic vortex of the accuracy study, 128^2 p = 3 with CFL
        # steps: a state that stays in L2, in both precisions
        _case("vortex_128_p3_f32", steps=64),
        _case("vortex_128_p3_f64", dtype="f64", steps=12),
        # the paper's own setting: Lobatto points and the chain-rule divergence
        _case("paper_128_p3_f32", pts="lobatto", div="chain", steps=64),
        # a production-size smooth solve, every array larger than L2
        _case("vortex_1024_p3_f32", nx=1024, ny=1024, steps=8),
        # the other orders at that number of unknowns, on odd, ragged grids
        _case("vortex_821x819_p4_f32", nx=821, ny=819, p=4, steps=6),
        _case("vortex_1365x1363_p2_f32", nx=1365, ny=1363, p=2, steps=6),
        # the discontinuous workload: four-quadrant Riemann problem with the
        # TVB limiter after every stage, transmissive boundaries
        _case("quadrant_512_p2_limited_f32", problem="quadrant", nx=512, ny=512, p=2, limiter=True, steps=12),
        # the finite-volume comparison scheme at the same number of unknowns
        _case("quadrant_1536_fv2_f32", problem="quadrant", scheme="fv2", nx=1536, ny=1536, p=0, steps=12),
        # gradient of a misfit through a rollout: forward with checkpoints,
        # recomputation and transposed steps
        _case("gradient_256_p3_f32", kind="rollout", nx=256, ny=256, steps=20, fixed=True),
        # the largest single-GPU workload: 64 ragged vortex solves of order 2-4
        # advanced together, autotuned
        {"name": "batch_64_f32", "kind": "batch", "dtype": "f32", "count": 64, "draw": 0, "lo": 32, "hi": 256,
         "steps": 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rate(c):
    """Rough unknown-stages per second, to keep a drawn pass within bounds."""
    if c.get("kind") == "rollout":
        return 6e9 if c["dtype"] == "f32" else 4e8
    return 3e10 if c["dtype"] == "f32" else 1.5e9


def draw(rng):
    kind = rng.choice(["step", "step", "step", "paper", "advection", "limited", "fv", "residual", "rollout", "batch"])
    if kind == "batch":
        return {"kind": "batch", "dtype": "f32", "count": rng.randint(3, 40), "draw": rng.randrange(1, 10000),
                "lo": 24, "hi": rng.randint(64, 256), "steps": rng.randint(1, 20)}
    dtype = rng.choice(["f32", "f32", "f64"])
    top = 1024 if dtype == "f32" else 400
    nx = _log_int(rng, 16, top)
    ny = max(9, min(top, int(round(nx * math.exp(rng.uniform(-0.5, 0.5))))))
    c = _case(nx=nx, ny=ny, p=rng.randint(1, 4), dtype=dtype)
    if kind == "residual":
        c.update(kind="residual", steps=0, flux=rng.choice(["rusanov", "roe"]), corr=rng.choice(["gdg", "ndg"]))
        return c
    if kind == "paper":
        c.update(pts="lobatto", div="chain", flux=rng.choice(["rusanov", "roe"]))
    elif kind == "advection":
        c.update(problem="sine", flux=rng.choice(["rusanov", "upwind"]), fixed=True)
    elif kind == "limited":
        c.update(problem="quadrant", limiter=True, p=rng.randint(1, 3))
    elif kind == "fv":
        c.update(problem="quadrant", scheme=rng.choice(["fv2", "fv3"]), nx=min(1536, 3 * nx), ny=min(1536, 3 * ny), p=0)
    elif kind == "rollout":
        c.update(kind="rollout", fixed=True, nx=min(nx, 300), ny=min(ny, 300))
    else:
        c.update(fixed=rng.random() < 0.3)
    dof = c["nx"] * c["ny"] * (c["p"] + 1) ** 2
    most = int(0.03 * _rate(c) / (3 * dof))  # a pass of at most about 30 ms
    cap = 10 if kind == "limited" else 24 if kind == "rollout" else 100
    c["steps"] = max(1, min(_log_int(rng, 1, cap), most))
    return c


# ---------------------------------------------------------------------------
# problems (coordinates, initial states), 64-bit torch on the GPU
# ---------------------------------------------------------------------------
def _domain(c):
    return {"vortex": (0.0, 10.0, 0.0, 10.0), "sine": (0.0, 1.0, 0.0, 1.0), "quadrant": (0.0, 1.0, 0.0, 1.0)}[c["problem"]]


def _sizes(c):
    x0, x1, y0, y1 = _domain(c)
    return (x1 - x0) / c["nx"], (y1 - y0) / c["ny"]


def _nodes(n, pts):
    """Solution points and quadrature weights on [-1, 1]."""
    if n == 1:
        return np.zeros(1), np.full(1, 2.0)
    if pts == "gauss":
        return np.polynomial.legendre.leggauss(n)
    p = np.polynomial.legendre.Legendre.basis(n - 1)
    x = np.concatenate(([-1.0], np.sort(p.deriv().roots().real), [1.0]))
    return x, 2.0 / (n * (n - 1) * p(x) ** 2)


def _coords(c):
    """x, y of shape (ny, nx, n, n) broadcastable, [j, i, b, a]."""
    x0, _, y0, _ = _domain(c)
    hx, hy = _sizes(c)
    xi = torch.tensor(_nodes(c["p"] + 1, c["pts"])[0], dtype=torch.float64, device="cuda")
    ex = torch.arange(c["nx"], dtype=torch.float64, device="cuda")
    ey = torch.arange(c["ny"], dtype=torch.float64, device="cuda")
    x = x0 + hx * (ex[:, None] + 0.5 * (xi + 1.0))[None, :, None, :]
    y = y0 + hy * (ey[:, None] + 0.5 * (xi + 1.0))[:, None, :, None]
    return x, y


def _conserved(rho, u, v, p):
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])


def _vortex(x, y, eps, xc, yc, u0, v0):
    xb, yb = x - xc, y - yc
    xb, yb = xb - 10.0 * torch.floor(xb / 10.0 + 0.5), yb - 10.0 * torch.floor(yb / 10.0 + 0.5)
    r2 = xb * xb + yb * yb
    amp = eps / (2 * math.pi) * torch.exp(0.5 * (1.0 - r2))
    temp = 1.0 - (GAMMA - 1.0) * eps * eps / (8.0 * GAMMA * math.pi ** 2) * torch.exp(1.0 - r2)
    rho = temp ** (1.0 / (GAMMA - 1.0))
    return _conserved(rho, u0 - amp * yb, v0 + amp * xb, rho * temp)


def _initial(c, seed, which=0):
    """Initial state (V, ny * nx, n * n) of the case's type."""
    rng = np.random.default_rng([seed, which])
    n = c["p"] + 1
    x, y = _coords(c)
    if c["problem"] == "sine":
        a, b = rng.uniform(0.0, 1.0, 2)
        q = (rng.uniform(0.5, 1.5) * torch.sin(2 * math.pi * (x + a)) * torch.sin(2 * math.pi * (y + b)))[None]
    elif c["problem"] == "vortex":
        eps, xc, yc = c.get("eps", rng.uniform(3.0, 5.0)), *rng.uniform(3.0, 7.0, 2)
        q = _vortex(x, y, eps, xc, yc, *rng.uniform(0.8, 1.2, 2))
    else:
        # the four-quadrant states, split near (0.8, 0.8) on an element edge, pressures scaled
        s = rng.uniform(0.9, 1.1)
        sx, sy = (round(rng.uniform(0.7, 0.85) * c[k]) / c[k] for k in ("nx", "ny"))
        right, up = (x > sx).expand(c["ny"], c["nx"], n, n), (y > sy).expand(c["ny"], c["nx"], n, n)

        def pick(ur, ul, ll, lr):
            top = torch.where(right, ur, ul)
            low = torch.where(right, lr, ll)
            return torch.where(up, top, low).double()
        q = _conserved(pick(1.5, 0.5323, 0.138, 0.5323), pick(0.0, 1.206, 1.206, 0.0), pick(0.0, 0.0, 1.206, 1.206),
                       s * pick(1.5, 0.3, 0.029, 0.3))
    q = q.expand(q.shape[0], c["ny"], c["nx"], n, n).reshape(q.shape[0], c["ny"] * c["nx"], n * n)
    return q.to(torch.float32 if c["dtype"] == "f32" else torch.float64).contiguous()


def _config(c):
    x0, x1, y0, y1 = _domain(c)
    bc = nat.TRANSMISSIVE if c["problem"] == "quadrant" else nat.PERIODIC
    return nat.Config(eqn=nat.ADVECTION if c["problem"] == "sine" else nat.EULER, nx=c["nx"], ny=c["ny"],
                      x0=x0, x1=x1, y0=y0, y1=y1, p=c["p"], pts=PTS[c["pts"]], corr=CORR[c["corr"]],
                      flux=FLUX[c["flux"]], div=DIV[c["div"]], bc_x=bc, bc_y=bc, limiter=int(c["limiter"]),
                      tvb_M=50.0, lim_eps=1e-3, dtype=nat.F32 if c["dtype"] == "f32" else nat.F64,
                      cfl=CFL[c["p"]], scheme=SCHEME[c["scheme"]])


def _dt(c):
    """Fixed step size (0: CFL steps)."""
    if not c["fixed"]:
        return 0.0
    h = min(_sizes(c))
    if c["problem"] == "sine":
        return 1.0 / 227 if (c["nx"], c["ny"], c["p"]) == (16, 16, 2) else CFL[c["p"]] * h / math.sqrt(2.0)
    return CFL[c["p"]] * h / 4.0


def _instances(c):
    """Single cases of a batch: grid, order and vortex strength drawn once."""
    rng = np.random.default_rng(c["draw"])
    n = rng.integers(c["lo"], c["hi"] + 1, size=c["count"])
    p = rng.integers(2, 5, size=c["count"])
    eps = rng.uniform(1.0, 5.0, size=c["count"])
    return [_case(nx=int(n[k]), ny=int(n[k]), p=int(p[k]), dtype=c["dtype"], eps=float(eps[k]), steps=c["steps"])
            for k in range(c["count"])]


# ---------------------------------------------------------------------------
# the pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    if case["kind"] == "batch":
        single = _instances(case)
        q0 = [_initial(s, seed, k) for k, s in enumerate(single)]
        batch = nat.Batch([_config(s) for s in single])
        qs = [q.clone() for q in q0]
        batch.tune(qs)
        return {"case": case, "batch": batch, "q0": q0, "qs": qs}
    q0 = _initial(case, seed)
    state = {"case": case, "ctx": nat.Context(_config(case)), "q0": q0, "dt": _dt(case)}
    if case["kind"] == "residual":
        state["r"] = torch.empty_like(q0)
    elif case["kind"] == "rollout":
        state["target"] = _initial(case, seed, 1)
        state["weights"] = adjoint.quadrature_weights(state["ctx"])
    else:
        state["q"] = torch.empty_like(q0)
    return state


def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        for q, q0 in zip(state["qs"], state["q0"]):
            q.copy_(q0)
        return state["batch"].step(state["qs"], c["steps"])
    ctx = state["ctx"]
    if c["kind"] == "residual":
        return ctx.residual(state["q0"], state["r"])
    if c["kind"] == "rollout":
        q0 = state["q0"].detach().requires_grad_(True)
        q = adjoint.rollout(q0, ctx, c["steps"], state["dt"], 10)
        loss = 0.5 * (state["weights"] * (q - state["target"]) ** 2).sum()
        loss.backward()
        return {"q": q.detach(), "loss": loss.detach(), "grad": q0.grad}
    q = state["q"].copy_(state["q0"])
    if c["limiter"]:
        ctx.limit(q)
    return ctx.step(q, c["steps"], state["dt"])


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _stage_flops(c):
    """Operations per unknown and stage: point fluxes, line operators of both
    directions, corrections and a share of the common fluxes."""
    n = c["p"] + 1
    if c["problem"] == "sine":
        return 4 * n + 14
    return 25 + 16 * n + 32 + 240 // n


def work(case):
    """One SSP-RK3 stage reads its input state and writes its output, and
    stages 2 and 3 also read the state at the start of the step: 8 state
    arrays per step.  A transposed stage reads the state and the cotangent and
    writes the new one: 9 arrays per step."""
    if case["kind"] == "batch":
        parts = [work(s) for s in _instances(case)]
        return {k: sum(w[k] for w in parts) for k in ("bytes", "flops")}
    dof = case["nx"] * case["ny"] * (case["p"] + 1) ** 2
    array = dof * (1 if case["problem"] == "sine" else 4) * (4 if case["dtype"] == "f32" else 8)
    fl = _stage_flops(case) * dof
    if case["kind"] == "residual":
        return {"bytes": 2 * array, "flops": fl}
    if case["kind"] == "rollout":  # forward, recomputation, transposed steps
        return {"bytes": case["steps"] * array * (8 + 8 + 9), "flops": case["steps"] * fl * (3 + 3 + 6)}
    extra = 3 * array if case["limiter"] else 0  # the limiter reads every stage result
    return {"bytes": case["steps"] * (8 * array + extra), "flops": case["steps"] * 3 * fl}


# ---------------------------------------------------------------------------
# the same pass in plain 64-bit torch
# ---------------------------------------------------------------------------
class _Exact:
    """The semi-discrete scheme on q[v, j, i, b, a] in 64 bits."""

    def __init__(self, c):
        self.c = c
        self.hx, self.hy = _sizes(c)
        self.euler = c["problem"] != "sine"
        self.wall = c["problem"] == "quadrant"
        n = c["p"] + 1
        x, w = _nodes(n, c["pts"])
        P = np.polynomial.polynomial.Polynomial
        basis = []
        for l in range(n):
            poly = P([1.0])
            for m in range(n):
                if m != l:
                    poly = poly * P([-x[m], 1.0]) / (x[l] - x[m])
            basis.append(poly)
        D = np.array([[b.deriv()(xa) for b in basis] for xa in x])
        leg = np.polynomial.legendre.Legendre.basis
        # right Radau polynomial: 1 at -1, 0 at +1; its mirror image the other way round
        gl = (-1.0) ** n * 0.5 * (leg(n) - leg(n - 1))
        dgl = gl.deriv()(x)
        t = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")  # noqa: E731
        self.D, self.lm, self.lp = t(D), t([b(-1.0) for b in basis]), t([b(1.0) for b in basis])
        self.dgl, self.dgr = t(dgl), t(-gl.deriv()(-x))
        self.w2, self.xi = t(np.outer(w, w) / 4.0), t(x)

    # -- physics; d: 0 along x, 1 along y ---------------------------------
    def prim(self, q):
        u, v = q[1] / q[0], q[2] / q[0]
        return u, v, (GAMMA - 1.0) * (q[3] - 0.5 * (q[1] * u + q[2] * v))

    def flux(self, q, d):
        if not self.euler:
            return q
        u, v, p = self.prim(q)
        if d == 0:
            return torch.stack([q[1], q[1] * u + p, q[2] * u, (q[3] + p) * u])
        return torch.stack([q[2], q[1] * v, q[2] * v + p, (q[3] + p) * v])

    def jvp(self, q, dq, d):
        if not self.euler:
            return dq
        u, v, p = self.prim(q)
        vn, m = (u, 1) if d == 0 else (v, 2)
        dvn = (dq[m] - vn * dq[0]) / q[0]
        dp = (GAMMA - 1.0) * (dq[3] - (u * dq[1] + v * dq[2]) + 0.5 * (u * u + v * v) * dq[0])
        out = [dq[m], dq[1] * vn + q[1] * dvn, dq[2] * vn + q[2] * dvn, (dq[3] + dp) * vn + (q[3] + p) * dvn]
        out[m] = out[m] + dp
        return torch.stack(out)

    def common(self, a, b, d):
        """Common flux between the lower state a and the upper state b."""
        if not self.euler:
            return a  # both velocities are 1: Rusanov and upwind agree
        (ua, va, pa), (ub, vb, pb) = self.prim(a), self.prim(b)
        ca, cb = torch.sqrt(GAMMA * pa / a[0]), torch.sqrt(GAMMA * pb / b[0])
        na, nb = (ua, ub) if d == 0 else (va, vb)
        mean = 0.5 * (self.flux(a, d) + self.flux(b, d))
        if self.c["flux"] != "roe":
            sa, sb = na.abs() + ca, nb.abs() + cb
            return mean - 0.5 * torch.where(sa >= sb, sa, sb) * (b - a)
        wa, wb = torch.sqrt(a[0]), torch.sqrt(b[0])
        avg = lambda s, t: (wa * s + wb * t) / (wa + wb)  # noqa: E731
        rho, u, v, H = wa * wb, avg(ua, ub), avg(va, vb), avg((a[3] + pa) / a[0], (b[3] + pb) / b[0])
        c2 = (GAMMA - 1.0) * (H - 0.5 * (u * u + v * v))
        cs = torch.sqrt(c2)
        vn, vt = (u, v) if d == 0 else (v, u)
        dvt = vb - va if d == 0 else ub - ua
        dvn, dp = nb - na, pb - pa

        def fix(lam, lo, hi):  # Harten-Hyman
            e = torch.clamp(torch.maximum(lam - lo, hi - lam), min=0.0)
            return torch.where(lam.abs() < e, (lam * lam + e * e) / torch.where(e > 0, 2 * e, torch.ones_like(e)), lam.abs())
        l1, l4, l2 = fix(vn - cs, na - ca, nb - cb), fix(vn + cs, na + ca, nb + cb), vn.abs()
        a1, a4 = (dp - rho * cs * dvn) / (2 * c2), (dp + rho * cs * dvn) / (2 * c2)
        a2, a3 = (b[0] - a[0]) - dp / c2, rho * dvt
        one, zero = torch.ones_like(u), torch.zeros_like(u)
        nx, ny = (1.0, 0.0) if d == 0 else (0.0, 1.0)
        r = [(l1 * a1, [one, u - cs * nx, v - cs * ny, H - vn * cs]), (l2 * a2, [one, u, v, 0.5 * (u * u + v * v)]),
             (l2 * a3, [zero, one * ny, one * nx, vt]), (l4 * a4, [one, u + cs * nx, v + cs * ny, H + vn * cs])]
        return mean - 0.5 * torch.stack([sum(k * vec[m] for k, vec in r) for m in range(4)])

    # -- CPR ------------------------------------------------------------------
    def direction(self, q, d):
        """The part of -R along one direction; q[v, j, i, l, a] has the line
        elements on axis 2 and the points of a line on the last axis."""
        f = self.flux(q, d)
        eL, eR = q @ self.lm, q @ self.lp
        if self.c["div"] == "lp":
            r, fL, fR = f @ self.D.T, f @ self.lm, f @ self.lp
        else:
            r, fL, fR = self.jvp(q, q @ self.D.T, d), self.flux(eL, d), self.flux(eR, d)
        upper = torch.roll(eL, -1, 2)
        first = None
        if self.wall:
            upper = torch.cat([upper[:, :, :-1], eR[:, :, -1:]], 2)
            first = self.common(eL[:, :, :1], eL[:, :, :1], d)
        F = self.common(eR, upper, d)
        low = torch.roll(F, 1, 2)
        if self.wall:
            low = torch.cat([first, low[:, :, 1:]], 2)
        return r + (low - fL)[..., None] * self.dgl + (F - fR)[..., None] * self.dgr

    def rhs(self, q):
        if self.c["scheme"] != "cpr":
            return self.fv(q)
        rx = self.direction(q, 0)
        ry = self.direction(q.permute(0, 2, 1, 4, 3), 1).permute(0, 2, 1, 4, 3)
        return -(2.0 / self.hx) * rx - (2.0 / self.hy) * ry

    # -- finite volumes -------------------------------------------------------
    @staticmethod
    def minmod(a, b):
        return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))

    def fv_line(self, q, d):
        """Flux difference along axis 2 of q[v, j, i]."""
        k = q.shape[2]
        at = torch.arange(-2, k + 2, device=q.device)
        e = q[:, :, at.clamp(0, k - 1) if self.wall else at % k]
        dm, dp = e[:, :, 1:-1] - e[:, :, :-2], e[:, :, 2:] - e[:, :, 1:-1]
        b = e[:, :, 1:-1]
        if self.c["scheme"] == "fv2":
            s = 0.5 * self.minmod(dm, dp)
            up, dn = b + s, b - s
        else:
            up = b + self.minmod(dm, 4 * dp) / 6 + self.minmod(dp, 4 * dm) / 3
            dn = b - self.minmod(dp, 4 * dm) / 6 - self.minmod(dm, 4 * dp) / 3
        F = self.common(up[:, :, :-1], dn[:, :, 1:], d)
        return F[:, :, 1:] - F[:, :, :-1]

    def fv(self, q):
        s = q[..., 0, 0]
        r = -self.fv_line(s, 0) / self.hx - self.fv_line(s.transpose(1, 2), 1).transpose(1, 2) / self.hy
        return r[..., None, None]

    # -- limiter ------------------------------------------------------------
    def limit(self, q):
        if not self.c["limiter"]:
            return q
        avg = (q * self.w2).sum((-1, -2))

        def diffs(axis):
            up, dn = torch.roll(avg, -1, axis), torch.roll(avg, 1, axis)
            k = avg.shape[axis]
            if self.wall:
                up = torch.cat([up.narrow(axis, 0, k - 1), avg.narrow(axis, k - 1, 1)], axis)
                dn = torch.cat([avg.narrow(axis, 0, 1), dn.narrow(axis, 1, k - 1)], axis)
            return up - avg, avg - dn

        bad = torch.zeros_like(avg[0], dtype=torch.bool)
        slopes = []
        for axis, h, edges in ((2, self.hx, ((q @ self.lp, 1.0), (q @ self.lm, -1.0))),
                               (1, self.hy, ((q.transpose(-1, -2) @ self.lp, 1.0), (q.transpose(-1, -2) @ self.lm, -1.0)))):
            c = self.minmod(*diffs(axis))
            slopes.append(c / h)
            for e, s in edges:
                dl = s * (e - avg[..., None])
                off = (dl - self.minmod(dl, c[..., None].expand_as(dl))).abs()
                bad |= ((off > 1e-3) & (dl.abs() > 50.0 * h * h)).any(-1).any(0)
        lin = avg[..., None, None] + (0.5 * self.hx * self.xi) * slopes[0][..., None, None] \
            + (0.5 * self.hy * self.xi)[:, None] * slopes[1][..., None, None]
        return torch.where(bad[None, ..., None, None], lin, q)

    # -- time stepping --------------------------------------------------------
    def dt(self, q):
        if self.c["fixed"]:
            return _dt(self.c)
        u, v, p = self.prim(q)
        s = (torch.sqrt(u * u + v * v) + torch.sqrt(GAMMA * p / q[0])).max()
        return CFL[self.c["p"]] * min(self.hx, self.hy) / s

    def step(self, q, dt):
        q1 = self.limit(q + dt * self.rhs(q))
        q2 = self.limit(0.75 * q + 0.25 * (q1 + dt * self.rhs(q1)))
        return self.limit(q / 3.0 + (2.0 / 3.0) * (q2 + dt * self.rhs(q2)))

    def shaped(self, q):
        n = self.c["p"] + 1
        return q.double().reshape(q.shape[0], self.c["ny"], self.c["nx"], n, n)

    def solve(self, q):
        x = self.limit(self.shaped(q))
        for _ in range(self.c["steps"]):
            x = self.step(x, self.dt(x))
        return x.reshape(q.shape)


def exact(case, seed):
    if case["kind"] == "batch":
        return [_Exact(s).solve(_initial(s, seed, k)) for k, s in enumerate(_instances(case))]
    ex = _Exact(case)
    q0 = _initial(case, seed)
    if case["kind"] == "residual":
        return ex.rhs(ex.shaped(q0)).reshape(q0.shape)
    if case["kind"] == "step":
        return ex.solve(q0)
    from torch.utils.checkpoint import checkpoint
    x0 = ex.shaped(q0).requires_grad_(True)
    x = x0
    for _ in range(case["steps"]):
        x = checkpoint(ex.step, x, _dt(case), use_reentrant=False)
    w = ex.w2.reshape(-1) * (ex.hx * ex.hy)
    loss = 0.5 * (w * (x.reshape(q0.shape) - _initial(case, seed, 1).double()) ** 2).sum()
    loss.backward()
    return {"q": x.detach().reshape(q0.shape), "loss": loss.detach(), "grad": x0.grad.reshape(q0.shape)}
