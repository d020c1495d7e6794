"""The work that users of this library have it do, as measurable cases.

A case is one call sequence of a user's program on a solver it keeps: put a state in (canonical FP64
coefficients on the device), advance it, take the state out. listed() holds the workloads of this
repository's configurations (the 1D Burgers run, the 1D Euler Riemann problem, the 2D four-quadrant
problem, the vortex of the accuracy tables, the served and the batched mixes); draw() gives more of
the same ranges. exact() is the method written out in torch at 64 bits, without the library.

A solve in the FP32 form hands its coefficients on as float32, the type of its stage arithmetic; an
FP64 solve hands on float64.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2407_19169_gb300 import _native as N

GAMMA, CFL = 1.4, 0.1
EQS = {"advection": N.EQ_ADVECTION, "burgers": N.EQ_BURGERS, "euler": N.EQ_EULER}
DEFAULTS = dict(kind="solve", dim=2, nx=64, ny=1, k=2, eq="euler", precision="fp32", basis="Q", bc="outflow",
                filter="jump", limiter=False, steps=16, T=0.0)


def _solve(**kw):
    return {**DEFAULTS, **kw}


def listed():
    return [
        # the paper's first test problem: 200 cells, degree 2, FP64, advanced to a time; three kernels
        # of a few microseconds per step, so latency is everything
        _solve(name="burgers1d_p2_200_f64", dim=1, nx=200, k=2, eq="burgers", bc="periodic", precision="fp64",
               T=0.1, steps=0),
        # the 1D Euler Riemann problem in both precisions
        _solve(name="euler1d_p3_65536_f64", dim=1, nx=65536, k=3, precision="fp64", steps=16),
        _solve(name="euler1d_p3_65536_f32", dim=1, nx=65536, k=3, steps=64),
        # the largest 1D instance of the batched mix, an odd size, with the positivity limiter
        _solve(name="euler1d_p2_1000003_f32_limiter", dim=1, nx=1000003, k=2, limiter=True, steps=32),
        # the headline: 2048 x 2048, Q2, four quadrants, FP32 form; and the plain FP64 path on a
        # sixteenth of its cells
        _solve(name="euler2d_q2_2048_f32", nx=2048, ny=2048, steps=8),
        _solve(name="euler2d_q2_512_f64", nx=512, ny=512, precision="fp64", steps=4),
        # served solves alone on the device, smallest and largest side, limiter on as the engine has it
        _solve(name="euler2d_q2_128_f32_limiter", nx=128, ny=128, limiter=True, steps=16),
        _solve(name="euler2d_q2_1024_f32_limiter", nx=1024, ny=1024, limiter=True, steps=8),
        # degree 3 on a ragged periodic mesh
        _solve(name="euler2d_q3_509x517_f32", nx=509, ny=517, k=3, bc="periodic", steps=8),
        # the accuracy tables' space: total degree 3, FP64, periodic, 160 x 160
        _solve(name="euler2d_p3_160_f64", nx=160, ny=160, k=3, basis="P", bc="periodic", precision="fp64", steps=8),
        # one round of the serving engine: several resident solves advanced a chunk of 16 steps
        dict(name="served_round_q2_f32", kind="batch", persistent=False, limiter=True, steps=16,
             solves="2,128,2,outflow;2,256,2,outflow;2,256,2,outflow;2,512,2,outflow;2,512,2,outflow"),
        # the uneven batch in one persistent launch per class: both dimensions, every degree
        dict(name="batch_uneven_persistent_f32", kind="batch", persistent=True, limiter=True, steps=20,
             solves="1,1000,1,outflow;1,30002,2,periodic;1,400000,3,outflow;1,5462,3,periodic;1,90100,1,outflow;"
                    "2,64,1,periodic;2,310,1,outflow;2,178,2,outflow;2,512,2,periodic;2,90,3,outflow;"
                    "2,214,3,periodic;2,402,3,outflow"),
    ]


def _spread(r, lo, hi):
    """Log-uniform whole number in [lo, hi]."""
    return int(round(math.exp(r.uniform(math.log(lo), math.log(hi)))))


def draw(r):
    what = r.random()
    if what < 0.2:
        solves = []
        for _ in range(r.randint(2, 10)):
            dim = r.choice((1, 2))
            n = 2 * (_spread(r, 1000, 400000) // 2) if dim == 1 else 2 * (_spread(r, 64, 400) // 2)
            solves.append("%d,%d,%d,%s" % (dim, n, r.randint(1, 3), r.choice(("outflow", "periodic"))))
        return dict(kind="batch", persistent=r.random() < 0.5, limiter=r.random() < 0.75, steps=r.randint(8, 20),
                    solves=";".join(solves))
    k, precision = r.randint(1, 3), r.choice(("fp64", "fp32", "fp32"))
    eq = r.choice(("euler", "euler", "euler", "euler", "burgers", "advection"))
    c = dict(k=k, precision=precision, eq=eq, bc=r.choice(("outflow", "periodic")),
             filter=r.choice(("jump", "jump", "jump", "jump", "global", "hybrid", "off")))
    c["limiter"] = eq == "euler" and c["filter"] == "jump" and r.random() < 0.5
    if what < 0.45:
        return _solve(dim=1, nx=_spread(r, 40, 100000 if precision == "fp64" else 1000000), steps=r.randint(8, 48), **c)
    side = 256 if precision == "fp64" else 1024
    return _solve(nx=_spread(r, 32, side), ny=_spread(r, 32, side), basis=r.choice("QQP"), steps=r.randint(4, 16), **c)


# ---- the solves of a case -------------------------------------------------------------------------


def _solves(case):
    """The case's solves, each a dict of DEFAULTS' keys."""
    if case["kind"] == "solve":
        return [_solve(**case)]
    out = []
    for text in case["solves"].split(";"):
        dim, n, k, bc = text.split(",")
        dim, n = int(dim), int(n)
        out.append(_solve(dim=dim, nx=n, ny=n if dim == 2 else 1, k=int(k), bc=bc, limiter=case["limiter"],
                          steps=case["steps"]))
    return out


def _box(c):
    """The mesh's extent: the paper's [0, 2] for 1D Burgers, [0, 10]^2 for periodic 2D, else unit."""
    if c["dim"] == 1:
        return 2.0 if c["eq"] == "burgers" else 1.0
    return 10.0 if c["bc"] == "periodic" else 1.0


def _nvars(c):
    return 1 if c["eq"] != "euler" else (3 if c["dim"] == 1 else 4)


def _modes(c):
    """(p, q) of each mode, q outer."""
    k = c["k"]
    if c["dim"] == 1:
        return [(p, 0) for p in range(k + 1)]
    return [(p, q) for q in range(k + 1) for p in range(k + 1) if c["basis"] == "Q" or p + q <= k]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _legendre(k, x):
    """P_l and P_l' at the points x, each [l, point]."""
    P, D = np.zeros((k + 1, len(x))), np.zeros((k + 1, len(x)))
    for l in range(k + 1):
        s = np.polynomial.legendre.Legendre.basis(l)
        P[l], D[l] = s(x), s.deriv()(x)
    return P, D


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=_device())


def _initial(c, seed):
    """Canonical coefficients [v, mode, cell] of seeded data: two or four constant states meeting at a
    face next to the middle (outflow) or one mean state (periodic), with waves from the domain's
    length down to sixteen cells on top; projected with k + 3 Gauss points per direction."""
    r = random.Random(seed * 1000003 + c["nx"] * 31 + c["ny"] * 17 + c["k"])
    k, n, L = c["k"], (c["nx"], c["ny"]), _box(c)
    two = c["dim"] == 2
    xg, wg = np.polynomial.legendre.leggauss(k + 3)
    P, _ = _legendre(k, xg)
    h = [L / n[0], L / n[1]]
    at = [_t((np.arange(m)[:, None] + 0.5 + 0.5 * xg[None]) * hh) for m, hh in zip(n, h)]   # [cell, point]
    X = at[0][None, None]                                                # [y, b, x, a]
    Y = at[1][:, :, None, None] if two else torch.zeros(1, 1, 1, 1, dtype=torch.float64, device=_device())
    gentle = c["bc"] == "periodic" or not c["limiter"]
    states = []
    for _ in range(4):
        lo, hi, speed = (0.7, 1.5, 0.4) if gentle else (0.1, 2.0, 1.0)
        states.append((r.uniform(lo, hi), r.uniform(-speed, speed), r.uniform(-speed, speed), r.uniform(lo, hi)))
    right = X > (n[0] // 2) * h[0]
    upper = (Y > (n[1] // 2) * h[1]) if two else torch.zeros_like(Y, dtype=torch.bool)
    prim = []
    for f in range(4):
        a, b, d, e = (s[f] for s in states)
        if c["bc"] == "periodic":
            base = torch.full((1, 1, 1, 1), a, dtype=torch.float64, device=_device())
        else:
            base = torch.where(right, torch.where(upper, a, e), torch.where(upper, b, d))
        wave = torch.zeros_like(X + Y)
        for _ in range(4):
            kx = _spread(r, 1, max(1, n[0] // 16))
            ky = _spread(r, 1, max(1, n[1] // 16)) if two else 0
            wave = wave + r.uniform(0.01, 0.03) * torch.sin(2 * math.pi / L * (kx * X + ky * Y) + r.uniform(0, 6.28))
        prim.append(base * (1 + wave) if f in (0, 3) else base + wave)
    if c["eq"] != "euler":
        U = [0.5 + prim[1] + (0.0 if c["bc"] == "outflow" else torch.sin(2 * math.pi / L * X + 0 * Y))]
    else:
        rho, u, v, p = prim
        if two:
            U = [rho, rho * u, rho * v, p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)]
        else:
            U = [rho, rho * u, p / (GAMMA - 1) + 0.5 * rho * u * u]
    wx = _t(P * wg * (np.arange(k + 1)[:, None] + 0.5))                    # [p, a]
    out = []
    for w in U:
        w = torch.einsum("ybxa,pa->pybx", w.expand(n[1] if two else 1, len(xg) if two else 1, n[0], len(xg)), wx)
        w = torch.einsum("pybx,qb->qpyx", w, wx) if two else w[:, :, 0].unsqueeze(0)
        out.append(torch.stack([w[q, p].reshape(-1) for p, q in _modes(c)]))
    return torch.stack(out)


def _solver(c, stream):
    kinds = {"global": N.FILTER_GLOBAL}
    L, bc = _box(c), N.BC_PERIODIC if c["bc"] == "periodic" else N.BC_OUTFLOW
    return N.Solver(dim=c["dim"], nx=c["nx"], ny=c["ny"], x0=0.0, x1=L, y0=0.0, y1=L, bc=(bc,) * 4, k=c["k"],
                    eq=EQS[c["eq"]], filter=int(c["filter"] != "off"), cfl=CFL, gamma=GAMMA, adv=(1.0, 0.5),
                    basis=N.BASIS_Q if c["basis"] == "Q" else N.BASIS_P,
                    precision=N.PREC_FP64 if c["precision"] == "fp64" else N.PREC_FP32_MIXED,
                    stream=stream.cuda_stream, positivity=int(c["limiter"]), hybrid=int(c["filter"] == "hybrid"),
                    filter_kind=kinds.get(c["filter"], N.FILTER_JUMP))


def prepare(case, seed):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        solves = _solves(case)
        start = [_initial(c, seed + 7919 * i) for i, c in enumerate(solves)]
        return {"case": case, "solves": solves, "stream": stream, "start": start,
                "out": [torch.empty_like(u) for u in start], "solvers": [_solver(c, stream) for c in solves]}


def run(state):
    case, solvers = state["case"], state["solvers"]
    with torch.cuda.stream(state["stream"]):
        for s, u in zip(solvers, state["start"]):
            s.write_state_device(u.data_ptr(), u.numel())
        if case["kind"] == "batch":
            N.batch_run(solvers, case["steps"], persistent=case["persistent"])
        elif case["T"]:
            solvers[0].advance_to(case["T"])
        else:
            solvers[0].advance_steps(case["steps"])
        times, states = [], []
        for c, s, u in zip(state["solves"], solvers, state["out"]):
            times.append(s.read_state_device(u.data_ptr(), u.numel()))
            states.append(u if c["precision"] == "fp64" else u.float())
    return {"t": times, "u": states}


def _steps(c):
    """Steps of a solve; for a run to a time, from the CFL condition at unit-order wave speeds."""
    return c["steps"] or int(c["T"] * 1.5 / (CFL * _box(c) / c["nx"]))


def work(case):
    """Bytes: the state in and out in FP64 (an FP32 result out in 4 bytes). Flops per cell and stage:
    the sum-factorised transforms, the fluxes and the filter's end derivatives."""
    nbytes = flops = 0.0
    for c in _solves(case):
        cells, nv, nm, k1 = c["nx"] * c["ny"], _nvars(c), len(_modes(c)), c["k"] + 1
        nbytes += cells * nv * nm * (16 if c["precision"] == "fp64" else 12)
        if c["dim"] == 1:
            per = 2 * nv * nm * (2 * k1 + 2 + k1) + (k1 + 2) * 25
        else:
            per = 2 * nv * nm * (2 * k1 + 2 * k1 + 8 + 4 * k1) + (k1 * k1 + 4 * k1) * 25
        flops += 3.0 * _steps(c) * cells * per
    return {"bytes": nbytes, "flops": flops}


# ---- the method at 64 bits ------------------------------------------------------------------------


def _primitive(U):
    """(velocities, pressure) of conservative Euler variables [v, ...]."""
    vel = [m / U[0] for m in U[1:-1]]
    return vel, (GAMMA - 1) * (U[-1] - 0.5 * sum(m * w for m, w in zip(U[1:-1], vel)))


def _flux(c, U, d):
    if c["eq"] == "advection":
        return (1.0, 0.5)[d] * U
    if c["eq"] == "burgers":
        return 0.5 * U * U
    vel, p = _primitive(U)
    F = U * vel[d]
    F[1 + d] += p
    F[-1] += vel[d] * p
    return F


def _speed(c, U, d):
    if c["eq"] == "advection":
        return torch.full_like(U[0], (1.0, 0.5)[d])
    if c["eq"] == "burgers":
        return U[0].abs()
    vel, p = _primitive(U)
    return vel[d].abs() + torch.sqrt(GAMMA * p / U[0])


class _Method:
    """SSP-RK3 discontinuous Galerkin steps with the jump filter. Coefficients [v, q, p, y, x], in 1D
    with one q and one y; total degree as zero coefficients."""

    def __init__(self, c):
        self.c, self.k, k = c, c["k"], c["k"]
        self.dims = c["dim"]
        self.h = [_box(c) / c["nx"], _box(c) / c["ny"]]
        xg, wg = np.polynomial.legendre.leggauss(k + 1)
        P, D = _legendre(k, xg)
        self.P, self.WP, self.WD = _t(P), _t(P * wg), _t(D * wg)
        self.sign = _t((-1.0) ** np.arange(k + 1))
        # end[l, r] = P_l^(r)(1)
        self.end = [[0.0 if r > l else float(np.polynomial.legendre.Legendre.basis(l).deriv(r)(1.0)) if r
                     else 1.0 for r in range(k + 1)] for l in range(k + 1)]
        kq = k + 1 if self.dims == 2 else 1
        l = torch.arange(k + 1, device=_device())
        self.degree = l[None, :] + l[:kq, None]                            # [q, p]
        self.keep = (self.degree <= k) | (c["basis"] == "Q")
        self.lmax = 2 * k if self.dims == 2 and c["basis"] == "Q" else k
        mids = [0.0] if k == 3 else []
        ends = [-1.0, 1.0]
        if self.dims == 1:
            pts = [(x, 0.0) for x in list(xg) + ends + mids]
        else:
            pts = [(x, y) for x in xg for y in xg] + [(x, e) for x in xg for e in ends + mids] + \
                  [(e, y) for y in xg for e in ends + mids]
        V = [_legendre(k, np.array([q[d] for q in pts]))[0] for d in (0, 1)]
        self.points = _t(np.einsum("qi,pi->iqp", V[1][:kq], V[0]))

    def beyond(self, lo, hi, ghost_lo, ghost_hi, d):
        """Face pairs along direction d from cell end values: lo/hi of each cell; the ghosts' values
        next to the first and last face (periodic: the cells across)."""
        ax = -1 - d
        if self.c["bc"] == "periodic":
            ghost_lo, ghost_hi = hi.narrow(ax, -1, 1), lo.narrow(ax, 0, 1)
        return torch.cat([ghost_lo, hi], ax), torch.cat([lo, ghost_hi], ax)

    def ghosts(self, U, shape, d):
        """The outflow ghosts' values: the averages of the first and last cells, in end values of
        `shape` coefficients per cell."""
        ax = -1 - d
        avg = U[:, 0, 0]
        return [avg.narrow(ax, i, 1).unsqueeze(1).expand(-1, shape, -1, -1) for i in (0, -1)]

    def moments(self, U, d):
        """Flux moments [v, l, faces...] of the faces normal to direction d."""
        A = U if d == 0 else U.transpose(1, 2)                              # [v, along the face, normal]
        hi, lo = A.sum(2), torch.einsum("vlnyx,n->vlyx", A, self.sign)
        if self.dims == 2:
            hi, lo = (torch.einsum("vlyx,lg->vgyx", e, self.P) for e in (hi, lo))
        a, b = self.beyond(lo, hi, *self.ghosts(U, hi.shape[1], d), d)
        alpha = torch.maximum(_speed(self.c, a, d), _speed(self.c, b, d))
        F = 0.5 * (_flux(self.c, a, d) + _flux(self.c, b, d) - alpha * (b - a))
        return torch.einsum("vgyx,lg->vlyx", F, self.WP) if self.dims == 2 else F

    def residual(self, U):
        k1 = self.k + 1
        two = self.dims == 2
        W = torch.einsum("vqpyx,pa->vqayx", U, self.P)
        if two:
            W = torch.einsum("vqayx,qb->vbayx", W, self.P)
        R = torch.zeros_like(U)
        l = torch.arange(k1, dtype=torch.float64, device=_device())
        norm = (2 * l[None] + 1) * (2 * l[:U.shape[1], None] + 1)
        for d in range(self.dims):
            F = _flux(self.c, W, d)
            V = torch.einsum("vbayx,pa->vbpyx", F, self.WD if d == 0 else self.WP)
            if two:
                V = torch.einsum("vbpyx,qb->vqpyx", V, self.WP if d == 0 else self.WD)
            M = self.moments(U, d)
            ax, n = -1 - d, U.shape[-1 - d]
            lo, hi = M.narrow(ax, 0, n), M.narrow(ax, 1, n)
            if d == 0:
                V += self.sign[None, None, :, None, None] * lo[:, :, None] - hi[:, :, None]
            else:
                V += self.sign[None, :, None, None, None] * lo[:, None] - hi[:, None]
            R += V * ((norm / (2 if two else 1)) / self.h[d])[None, :, :, None, None]
        return R * self.keep[None, :, :, None, None]

    def jumps(self, U, d):
        """Per total derivative order m: the sum over derivatives of order m of the faces' averaged
        absolute jumps, [v, faces...], physical derivatives."""
        k, two = self.k, self.dims == 2
        A = U if d == 0 else U.transpose(1, 2)
        S = [0.0] * (self.lmax + 1)
        for n in range(k + 1):                                              # derivatives across the face
            e = _t([self.end[l][n] for l in range(k + 1)])
            hi = torch.einsum("vlnyx,n->vlyx", A, e)
            lo = torch.einsum("vlnyx,n->vlyx", A, e * self.sign * (-1.0) ** n)
            g = [torch.zeros_like(x) for x in self.ghosts(U, hi.shape[1], d)]
            if n == 0:
                for x, y in zip(g, self.ghosts(U, 1, d)):
                    x[:, :1] = y
            a, b = self.beyond(lo, hi, *g, d)
            J = b - a
            for t in range(k + 1 if two else 1):                             # along the face
                if two and self.c["basis"] == "P" and n + t > k:
                    continue
                scale = (2 / self.h[d]) ** n * (2 / self.h[1 - d]) ** t
                if two:
                    e = _t([self.end[l][t] for l in range(k + 1)])
                    up = torch.einsum("vlyx,l->vyx", J, e)
                    down = torch.einsum("vlyx,l->vyx", J, e * self.sign)
                    S[n + t] = S[n + t] + 0.5 * scale * (up.abs() + down.abs())
                else:
                    S[n] = S[n] + scale * J[:, 0].abs()
        ax, cells = -1 - d, U.shape[-1 - d]
        return [s.narrow(ax, 0, cells) + s.narrow(ax, 1, cells) if torch.is_tensor(s) else s for s in S]

    def parameters(self, avg):
        beta = [_speed(self.c, avg, d) for d in range(self.dims)]
        if self.c["eq"] != "euler":
            return beta, 1.0
        return beta, avg[0] / (avg[-1] + _primitive(avg)[1])

    def damp(self, U, dt):
        """The filter (or the hybrid limiter) of one stage."""
        kind = self.c["filter"]
        if kind == "off":
            return U
        beta, inv_h = self.parameters(U[:, 0, 0])
        total, eta, factors = 0.0, 0.0, []
        S = [self.jumps(U, d) for d in range(self.dims)]
        for m in range(self.lmax + 1):
            for d in range(self.dims):
                w = 1.0 if m == 0 else m * (m + 1) * self.h[d] ** m
                scale = 1.0 if self.dims == 2 else 1.0 / self.h[0]
                total = total + beta[d] * scale * w * S[d][m]
                if m == 0:
                    eta = eta + S[d][0][0] / (2 * self.h[d])
            factors.append(torch.exp(-total.amax(0) * inv_h * dt))
        factors[0] = torch.ones_like(factors[0])
        if kind == "global":
            factors[1:] = [factors[-1]] * self.lmax
        factors = torch.stack(factors)
        if kind == "hybrid":
            top = eta.max()
            omega = torch.where(eta > 1, (top - eta) / (top - 1), 1.0)
            factors = omega + (1 - omega) * factors
        return U * factors[self.degree.clamp(max=self.lmax)]

    def values(self, U):
        return torch.einsum("iqp,vqpyx->viyx", self.points, U)

    def limit(self, U):
        """The positivity limiter: density, then pressure, scaled towards the averages."""
        avg = U[:, 0, 0]
        pbar = _primitive(avg)[1]
        low_r = 1e-3 * avg[0]
        low_p = torch.minimum(torch.minimum(1e-3 * (avg[0] + avg[-1].abs()), avg[0]), pbar)
        rmin = torch.minimum(torch.einsum("iqp,qpyx->iyx", self.points, U[0]).amin(0), avg[0])
        theta = torch.where(rmin < low_r, (avg[0] - low_r) / (avg[0] - rmin), 1.0)
        U = U.clone()
        high = U[0].clone()
        U[0] *= theta
        U[0, 0, 0] = high[0, 0]
        W = self.values(U)
        bad = _primitive(W)[1] < low_p
        cells = bad.any(0).nonzero(as_tuple=True)
        if len(cells[0]):
            w, a, low, b = W[:, :, cells[0], cells[1]], avg[:, None, cells[0], cells[1]], low_p[cells], bad[:, cells[0], cells[1]]
            lo, hi = torch.zeros_like(w[0]), torch.ones_like(w[0])
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                ok = _primitive(a + mid * (w - a))[1] >= low
                lo, hi = torch.where(ok, mid, lo), torch.where(ok, hi, mid)
            t = torch.where(b, lo, 1.0).amin(0)
            part = U[:, :, :, cells[0], cells[1]] * t
            part[:, 0, 0] = a[:, 0]
            U[:, :, :, cells[0], cells[1]] = part
        return U

    def rate(self, U):
        at = [U[:, 0, 0]] + ([self.values(U)] if self.c["limiter"] else [])
        return max(float(sum(_speed(self.c, w, d) / self.h[d] for d in range(self.dims)).max()) for w in at)

    def step(self, U, dt):
        V = U
        for c0, c1 in ((0.0, 1.0), (0.75, 0.25), (1 / 3, 2 / 3)):
            V = self.damp(c0 * U + c1 * (V + dt * self.residual(V)), dt)
            if self.c["limiter"]:
                V = self.limit(V)
        return V


def _advance(c, u):
    modes = _modes(c)
    U = torch.zeros(_nvars(c), c["k"] + 1 if c["dim"] == 2 else 1, c["k"] + 1, c["ny"], c["nx"], dtype=torch.float64,
                    device=_device())
    for m, (p, q) in enumerate(modes):
        U[:, q, p] = u[:, m].reshape(-1, c["ny"], c["nx"])
    method, t, n = _Method(c), 0.0, 0
    end = c["T"] or math.inf
    while t < end and (c["T"] or n < c["steps"]):
        dt = CFL / method.rate(U)
        last = t + dt >= end
        dt = end - t if last else dt
        U = method.step(U, dt)
        t, n = (end if last else t + dt), n + 1
    return torch.stack([U[:, q, p].reshape(_nvars(c), -1) for p, q in modes], 1), t


def exact(case, seed):
    done = [_advance(c, _initial(c, seed + 7919 * i)) for i, c in enumerate(_solves(case))]
    return {"t": [t for _, t in done], "u": [u for u, _ in done]}
