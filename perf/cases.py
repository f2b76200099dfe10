"""Timed cases: the calls a user of the solver makes, over the sizes, precisions
and equations that the package is used at.

A case says which call is made (``call``), on which problem (``problem``), at
which size and precision, and for how many steps:

  step        Solver.step, the plain call, with the default options
  persistent  Solver.run_persistent, K steps of a 1D batch in one launch
              (``cluster``: the cluster form for a few small instances)
  graph       Solver.run_graph, K steps as a CUDA graph
  rhs         Solver.rhs, the spatial operator alone
  adjoint     Solver.step_record and the adjoint of that step
  gradient    adjoint.run_to_time, a run and its gradient

``exact`` evaluates the same scheme with plain torch operations in 64 bits
(the paper's formulas as printed, gradients by torch.autograd).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2207_05258_gb300 import hweno
from paper_2207_05258_gb300.adjoint import run_to_time

GAMMA = 1.4
# operations of the scheme as printed, per point and step (counted)
FLOPS = {("euler", 1): 4870.2, ("burgers", 1): 1198.1, ("buckley", 1): 1296.3,
         ("euler", 2): 14555.8, ("burgers", 2): 2484.8}
# the same of one forward-mode step (values and tangents): an adjoint step
ADJOINT_FLOPS = {("euler", 2): 45603.2, ("burgers", 1): 3722.2}

EQUATION = {"burgers": "burgers", "riemann": "euler", "blast": "euler", "buckley": "buckley",
            "burgers2d": "burgers", "wave2d": "euler", "mach2d": "euler"}


def _case(name, call, problem, precision="fp64", sizes="", count=1, nx=0, ny=0, steps=1,
          cluster=False):
    c = dict(name=name, call=call, problem=problem, precision=precision, sizes=sizes,
             count=count, nx=nx, ny=ny, steps=steps, cluster=cluster)
    if not name:
        del c["name"]
    return c


def listed():
    return [
        _case("burgers_400_cluster", "persistent", "burgers", sizes="400", steps=20, cluster=True),
        _case("riemann_200_step", "step", "riemann", sizes="200"),
        _case("blast_800_cluster", "persistent", "blast", sizes="800", steps=10, cluster=True),
        _case("riemann_batch_fp64", "persistent", "riemann", sizes="200,400,800,1600,3200",
              count=2048, steps=2),
        _case("riemann_batch_fp32", "graph", "riemann", "fp32", sizes="200,400,800,1600,3200",
              count=2048, steps=8),
        _case("buckley_batch_fp64", "persistent", "buckley", sizes="187,401,1333", count=384,
              steps=4),
        _case("wave2d_256_fp64", "step", "wave2d", nx=256, ny=256, steps=2),
        _case("mach2d_1920_fp64", "step", "mach2d", nx=1920, ny=480, steps=1),
        _case("wave2d_1024_fp32", "graph", "wave2d", "fp32", nx=1024, ny=1024, steps=4),
        _case("burgers2d_rhs_fp64", "rhs", "burgers2d", nx=321, ny=203),
        _case("wave2d_256_adjoint", "adjoint", "wave2d", nx=256, ny=256),
        _case("burgers_gradient", "gradient", "burgers", sizes="800", count=256, steps=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "batch", "batch", "grid", "grid", "rhs", "adjoint", "gradient"])
    precision = rng.choice(["fp64", "fp64", "fp32"])
    if kind == "small":
        call = rng.choice(["step", "persistent"])
        return _case("", call, rng.choice(["burgers", "riemann", "blast"]),
                     sizes=str(_log_int(rng, 40, 992)), cluster=call == "persistent",
                     steps=1 if call == "step" else rng.randint(5, 20))
    if kind == "batch":
        sizes = sorted({_log_int(rng, 60, 3200) for _ in range(rng.randint(1, 5))})
        points = _log_int(rng, 2e4, 2.5e6)
        return _case("", "graph" if precision == "fp32" else "persistent",
                     rng.choice(["riemann", "riemann", "buckley", "burgers"]), precision,
                     sizes=",".join(str(n) for n in sizes),
                     count=max(1, points * len(sizes) // sum(sizes)), steps=rng.randint(1, 2))
    if kind == "grid":
        problem = rng.choice(["wave2d", "mach2d", "burgers2d"])
        nx = _log_int(rng, 48, 1400)
        ny = max(48, nx // 4) if problem == "mach2d" else _log_int(rng, 48, 640)
        return _case("", rng.choice(["step", "graph"]), problem, precision, nx=nx, ny=ny,
                     steps=1 if nx * ny > 300000 else rng.randint(1, 4))
    if kind == "rhs":
        if rng.random() < 0.5:
            return _case("", "rhs", rng.choice(["burgers2d", "wave2d"]), precision,
                         nx=_log_int(rng, 48, 1000), ny=_log_int(rng, 48, 640))
        return _case("", "rhs", "riemann", precision, sizes=str(_log_int(rng, 60, 3200)),
                     count=_log_int(rng, 1, 512))
    if kind == "adjoint":
        return _case("", "adjoint", "wave2d", nx=_log_int(rng, 40, 400), ny=_log_int(rng, 40, 400))
    return _case("", "gradient", "burgers", sizes=str(_log_int(rng, 80, 1600)),
                 count=_log_int(rng, 1, 256), steps=rng.randint(2, 6))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _centers(lo, hi, n):
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    return lo + (i + 0.5) * ((hi - lo) / n)


def _sizes(case):
    s = [int(x) for x in case["sizes"].split(",")]
    return [s[k % len(s)] for k in range(case["count"])]


def _euler1d(r, u, p, dr, du, dp):
    U = torch.stack([r, r * u, p / (GAMMA - 1) + 0.5 * r * u * u], 1)
    V = torch.stack([dr, dr * u + r * du, dp / (GAMMA - 1) + 0.5 * dr * u * u + r * u * du], 1)
    return U, V


def _states1d(problem, n, z):
    """(U, V), each [B][m][n], of the instances whose random numbers are the
    rows of z (uniform in [0, 1), 16 per instance)."""
    z = torch.from_numpy(np.ascontiguousarray(z)).cuda()
    c = lambda k, lo=0.0, hi=1.0: (lo + (hi - lo) * z[:, k])[:, None]  # noqa: E731
    if problem == "burgers":
        # Examples 3.1 and 3.3, four Fourier modes more and a jump that a
        # third of the instances have
        x = _centers(0.0, 2.0, n)[None]
        U, V = 0.5 + torch.sin(math.pi * x), math.pi * torch.cos(math.pi * x)
        for k in range(1, 5):
            a, ph = c(k, -0.05, 0.05), c(4 + k, 0.0, 2 * math.pi)
            U = U + a * torch.sin(k * math.pi * x + ph)
            V = V + a * k * math.pi * torch.cos(k * math.pi * x + ph)
        U = U + torch.where((c(9) < 1.0 / 3.0) & (x > c(10, 0.4, 1.6)), c(11, -0.6, 0.6), 0.0)
        return U[:, None], V[:, None]
    if problem == "buckley":  # Example 3.4
        x = _centers(-1.0, 1.0, n)[None]
        inside = (x >= c(1, -0.6, -0.4)) & (x <= c(2, -0.1, 0.1))
        U = torch.where(inside, c(0, 0.8, 1.0), 0.0)
        return U[:, None], torch.zeros_like(U)[:, None]
    x = _centers(0.0, 1.0, n)[None]
    zero = torch.zeros(z.shape[0], n, dtype=torch.float64, device="cuda")
    if problem == "blast":  # Example 3.7
        p = torch.where(x < 0.1, c(0, 800.0, 1200.0), torch.where(x < 0.9, c(1, 0.01, 0.02),
                                                                  c(2, 80.0, 120.0)))
        return _euler1d(zero + 1.0, zero, p + zero, zero, zero, zero)
    # Riemann problems, half of them running into a density wave (Example 3.6)
    left = x < 0.5
    pick = lambda a, b: torch.where(left, a, b) + zero  # noqa: E731
    r = pick(c(0, 0.1, 1.0), c(1, 0.1, 1.0))
    u = pick(c(2, -0.5, 0.5), c(3, -0.5, 0.5))
    p = pick(c(4, 0.1, 1.0), c(5, 0.1, 1.0))
    a = torch.where(c(6) < 0.5, c(7, 0.0, 0.3), 0.0) * c(1, 0.1, 1.0)
    k = 2 * math.pi * torch.floor(c(8, 1.0, 9.0))
    r = r + torch.where(left, 0.0, a * torch.sin(k * (x - 0.5)))
    dr = torch.where(left, 0.0, a * k * torch.cos(k * (x - 0.5)))
    return _euler1d(r, u, p, dr, zero, zero)


def _fourier2d(g, X, Y, kx, ky, amp):
    """A smooth field of four modes and its two derivatives."""
    f, fx, fy = torch.zeros_like(X), torch.zeros_like(X), torch.zeros_like(X)
    for _ in range(4):
        a, ph = amp / 4 * g.uniform(-1, 1), g.uniform(0, 2 * math.pi)
        i, j = kx * g.randint(0, 3), ky * g.randint(1, 3)
        s = i * X + j * Y + ph
        f, fx, fy = f + a * torch.sin(s), fx + a * i * torch.cos(s), fy + a * j * torch.cos(s)
    return f, fx, fy


MACH_POST = (8.0, 8.25 * math.cos(math.pi / 6), -8.25 * math.sin(math.pi / 6), 116.5)
MACH_PRE = (1.4, 0.0, 0.0, 1.0)


def _conserved2d(r, u, v, p):
    return (r, r * u, r * v, p / (GAMMA - 1) + 0.5 * r * (u * u + v * v))


def _grid(case):
    """Domain, boundary conditions and imposed states of the problem."""
    P = dict(x0=0.0, x1=1.0, y0=0.0, y1=1.0, bc=("periodic",) * 4, inflow=(0.0,) * 4,
             pre=(0.0,) * 4, dmr_x0=1.0 / 6.0, dmr_speed=10.0, dmr_angle=math.pi / 3)
    problem = case["problem"]
    if problem == "burgers":
        P["x1"] = 2.0
    elif problem == "buckley":
        P.update(x0=-1.0, bc=("outflow",) * 2 + ("periodic",) * 2)
    elif problem == "riemann":
        P["bc"] = ("outflow",) * 2 + ("periodic",) * 2
    elif problem == "blast":
        P["bc"] = ("reflective",) * 2 + ("periodic",) * 2
    elif problem == "burgers2d":
        P.update(x1=4.0, y1=4.0)
    elif problem == "wave2d":
        P.update(x1=2.0, y1=2.0)
    else:  # Example 3.11
        P.update(x1=4.0, bc=("inflow", "outflow", "dmr_bottom", "dmr_top"),
                 inflow=_conserved2d(*MACH_POST), pre=_conserved2d(*MACH_PRE))
    return P


def _fields(case, seed):
    """The initial U, V (, W), flat in the solver's layout, in the case's precision."""
    g = np.random.RandomState(seed % (1 << 32))
    if case["nx"] == 0:
        nx = _sizes(case)
        z = g.random_sample((len(nx), 16))
        rows = [None] * len(nx)
        for n in set(nx):
            who = [k for k, m in enumerate(nx) if m == n]
            U, V = _states1d(case["problem"], n, z[who])
            both = torch.stack([U.flatten(1), V.flatten(1)])
            for j, k in enumerate(who):
                rows[k] = both[:, j]
        U, V = torch.cat(rows, 1)
        fields = [U, V]
    else:
        P, nx, ny = _grid(case), case["nx"], case["ny"]
        Y, X = torch.meshgrid(_centers(P["y0"], P["y1"], ny), _centers(P["x0"], P["x1"], nx),
                              indexing="ij")
        kx, ky = 2 * math.pi / (P["x1"] - P["x0"]), 2 * math.pi / (P["y1"] - P["y0"])
        f, fx, fy = _fourier2d(g, X, Y, kx, ky, 0.05)
        if case["problem"] == "burgers2d":  # Examples 3.8 and 3.10
            s = 0.5 * math.pi * (X + Y)
            d = 0.5 * math.pi * torch.cos(s)
            fields = [(0.5 + torch.sin(s) + f)[None], (d + fx)[None], (d + fy)[None]]
        elif case["problem"] == "wave2d":  # Example 3.9 and smooth waves in every field
            s = math.pi * (X + Y)
            d = 0.2 * math.pi * torch.cos(s)
            q = [(1 + 0.2 * torch.sin(s) + f, d + fx, d + fy)]
            for mean in (0.7, 0.3, 1.0):
                a = _fourier2d(g, X, Y, kx, ky, 0.1)
                q.append((mean + a[0], a[1], a[2]))
            (r, u, v, p) = q
            out = [torch.stack(_conserved2d(r[0], u[0], v[0], p[0]))]
            for k in (1, 2):
                out.append(torch.stack([
                    r[k], r[k] * u[0] + r[0] * u[k], r[k] * v[0] + r[0] * v[k],
                    p[k] / (GAMMA - 1) + 0.5 * r[k] * (u[0] ** 2 + v[0] ** 2)
                    + r[0] * (u[0] * u[k] + v[0] * v[k])]))
            fields = out
        else:  # Example 3.11, a weak density wave over it
            post = X < 1.0 / 6.0 + Y / math.tan(math.pi / 3)
            r, u, v, p = (torch.where(post, a, b).to(torch.float64)
                          for a, b in zip(MACH_POST, MACH_PRE))
            e = 0.5 * (u * u + v * v)
            fields = [torch.stack(_conserved2d(r * (1 + f), u, v, p))]
            for k in (fx, fy):
                fields.append(torch.stack([r * k, r * k * u, r * k * v, r * k * e]))
    kind = torch.float32 if case["precision"] == "fp32" else torch.float64
    return [a.reshape(-1).to(kind) for a in fields]


def _cotangents(case, seed, fields):
    """Gradients of a functional with respect to the outputs: smooth and of order one."""
    g = np.random.RandomState((seed + 7919) % (1 << 32))
    out = []
    for a in fields:
        i = torch.arange(a.numel(), dtype=torch.float64, device="cuda")
        out.append(torch.sin(g.uniform(0.01, 0.05) * i + g.uniform(0, 6))
                   + 0.5 * torch.cos(g.uniform(0.001, 0.01) * i))
    return out


def _gradient_end(case):
    """A final time that instances reach in about case["steps"] steps."""
    return 0.6 * (2.0 / max(_sizes(case))) / 1.6 * case["steps"]


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case = case
    s.fields = _fields(case, seed)
    s.two = case["nx"] != 0
    P = _grid(case)
    size = dict(nx=case["nx"], ny=case["ny"]) if s.two else dict(nx=_sizes(case))
    if case["cluster"]:
        size["fused_small"] = 2
    s.solver = hweno.Solver(EQUATION[case["problem"]], 2 if s.two else 1, gamma=GAMMA,
                            precision=case["precision"], **P, **size)
    s.t = torch.zeros(s.solver.batch, dtype=torch.float64, device="cuda")
    s.work = [torch.empty_like(a) for a in s.fields]
    call = case["call"]
    if call in ("persistent", "graph") and not case["cluster"] or call == "step" and s.two:
        W = s.fields[2] if s.two else None
        s.solver.autotune(s.fields[0], s.fields[1], W, s.t, 1e30)
    if call == "graph":
        s.stream = torch.cuda.Stream()
    elif call == "adjoint":
        s.record, s.dt = s.solver.new_record(), torch.empty_like(s.t)
        s.t0 = torch.zeros_like(s.t)
        s.lam0 = _cotangents(case, seed, s.fields)
        s.lam = [torch.empty_like(a) for a in s.lam0]
    elif call == "gradient":
        s.lam0 = _cotangents(case, seed, s.fields)
        s.t_end = _gradient_end(case)
    torch.cuda.synchronize()
    return s


def _start(s):
    """The run's arrays from the initial data."""
    for a, b in zip(s.work, s.fields):
        a.copy_(b)
    s.t.zero_()
    return s.work + ([] if s.two else [None])


def run(s):
    call, steps = s.case["call"], s.case["steps"]
    if call == "rhs":
        return s.solver.rhs(s.fields[0], s.fields[1], s.fields[2] if s.two else None)
    if call == "gradient":
        U0, V0 = (a.clone().requires_grad_(True) for a in s.fields)
        U, V = run_to_time(U0, V0, s.solver, s.t_end, checkpoint_every=4,
                           max_steps=2 * s.case["steps"], check_every=s.case["steps"])
        torch.autograd.backward((U, V), tuple(s.lam0))
        return dict(U=U.detach(), V=V.detach(), gU=U0.grad, gV=V0.grad)
    if call == "adjoint":
        U, V, W = _start(s)
        for a, b in zip(s.lam, s.lam0):
            a.copy_(b)
        s.solver.step_record(U, V, W, s.t, 1e30, s.record, s.dt)
        s.solver.adjoint_step(*s.fields, s.dt, *s.lam, t=s.t0, record=s.record)
        return dict(U=U, V=V, W=W, gU=s.lam[0], gV=s.lam[1], gW=s.lam[2], t=s.t)
    if call == "graph":
        with torch.cuda.stream(s.stream):
            U, V, W = _start(s)
            s.solver.run_graph(U, V, W, s.t, 1e30, max_steps=steps, steps_per_launch=steps)
    elif call == "persistent":
        U, V, W = _start(s)
        s.solver.run_persistent(U, V, s.t, 1e30, steps, count=False)
    else:
        U, V, W = _start(s)
        for _ in range(steps):
            s.solver.step(U, V, W, s.t, 1e30)
    return dict(zip("UVW", s.work), t=s.t)


def work(case):
    two = case["nx"] != 0
    eq, dim = EQUATION[case["problem"]], 2 if two else 1
    points = case["nx"] * case["ny"] if two else sum(_sizes(case))
    m = (4 if two else 3) if eq == "euler" else 1
    word = 4 if case["precision"] == "fp32" else 8
    state = (3 if two else 2) * m * points * word
    flops = FLOPS[eq, dim] * points
    if case["call"] == "rhs":
        return dict(bytes=state + state + (2 if two else 1) * m * points * word, flops=flops / 3)
    if case["call"] == "adjoint":
        return dict(bytes=4 * state, flops=flops + ADJOINT_FLOPS[eq, dim] * points)
    if case["call"] == "gradient":
        return dict(bytes=4 * state,
                    flops=(flops + ADJOINT_FLOPS[eq, dim] * points) * case["steps"])
    return dict(bytes=2 * state, flops=flops * case["steps"])


# ---------------------------------------------------------------------------
# The scheme in plain torch, 64 bits. A field is a list of m tensors [L][n]:
# L lines (instances of one size, or the rows or columns of a grid) of n
# points along the direction of differentiation.
# ---------------------------------------------------------------------------
LIN_W = LIM_D = (0.98, 0.01, 0.01)
EPS, CFL = 1e-6, 0.6


def _sq(a):
    return a * a


def _weights(g, beta):
    tau = 0.25 * _sq((beta[0] - beta[1]).abs() + (beta[0] - beta[2]).abs())
    w = [g[k] * (1 + tau / (beta[k] + EPS)) for k in range(3)]
    s = w[0] + w[1] + w[2]
    return [a / s for a in w]


def _plus(f, h):
    """f-hat^+ at x_{i+1/2} from f and H = dx h at i-1, i, i+1 (Sec. 2.1)."""
    (fm, f0, fp), (hm, h0, hp) = f, h
    p0 = 11 / 60 * (fm + fp) + 19 / 30 * f0 + (hm + 10 * h0 - hp) / 20
    p1 = fm / 6 + 5 / 6 * f0 + 2 / 3 * h0
    p2 = 5 / 6 * f0 + fp / 6 + h0 / 3
    lap, dif = fm - 2 * f0 + fp, fm - fp
    a1 = 19 / 192 * (hm + hp) + 79 / 48 * h0 + 27 / 64 * dif
    a2 = 3 / 8 * (hm - hp) + 5 / 4 * lap
    a3 = -(11 / 24 * (hm + hp) + 17 / 6 * h0) - 15 / 8 * dif
    a4 = -(hm - hp) / 4 - lap / 2
    a5 = (hm + hp) / 4 + h0 + 3 / 4 * dif
    beta = [_sq(a1 + a3 / 4 + a5 / 16) + 13 / 3 * _sq(a2 + 63 / 130 * a4)
            + 781 / 20 * _sq(a3 + 8825 / 10934 * a5) + 1421461 / 2275 * _sq(a4)
            + 21520059541 / 1377684 * _sq(a5),
            _sq(h0) + 13 / 3 * _sq(h0 - f0 + fm), _sq(h0) + 13 / 3 * _sq(h0 + f0 - fp)]
    g = LIN_W
    w = _weights(g, beta)
    return w[0] * (p0 / g[0] - g[1] / g[0] * p1 - g[2] / g[0] * p2) + w[1] * p1 + w[2] * p2


def _derivative_plus(f, h):
    """dx p_0'(x_{i+1/2})."""
    return (f[0] - 8 * f[1] + 7 * f[2]) / 4 + (h[0] - 2 * h[1] - 5 * h[2]) / 12


def _limited(u, v, dx):
    """The limited derivative from u at i-1, i, i+1 and v at i-1, i+1 (Sec. 2.2)."""
    (um, u0, up), (vm, vp) = u, v
    q = [3 / (4 * dx) * (up - um) - (vm + vp) / 4, (u0 - um) / dx, (up - u0) / dx]
    a1 = -dx / 4 * (vm + vp) + 3 / 4 * (up - um)
    a2 = dx / 4 * (vm - vp) + um - 2 * u0 + up
    a3 = dx / 4 * (vm + vp) + (um - up) / 4
    a4 = dx / 4 * (vp - vm) - (um - 2 * u0 + up) / 2
    beta = [_sq(a1 + a3 / 4) + 13 / 3 * _sq(a2 + 63 / 130 * a4) + 781 / 20 * _sq(a3)
            + 1421461 / 2275 * _sq(a4), _sq(u0 - um), _sq(u0 - up)]
    d = LIM_D
    w = _weights(d, beta)
    return w[0] * (q[0] / d[0] - d[1] / d[0] * q[1] - d[2] / d[0] * q[2]) + w[1] * q[1] + w[2] * q[2]


def _primitive(U):
    """(velocities, p) of a list of conserved components."""
    vel = [a / U[0] for a in U[1:-1]]
    return vel, (GAMMA - 1) * (U[-1] - 0.5 * sum(a * b for a, b in zip(U[1:-1], vel)))


def _flux(eq, d, U):
    if eq == "burgers":
        return [0.5 * U[0] * U[0]]
    if eq == "buckley":
        return [4 * U[0] ** 2 / (4 * U[0] ** 2 + (1 - U[0]) ** 2)]
    vel, p = _primitive(U)
    F = [U[1 + d]] + [U[1 + d] * a for a in vel] + [(U[-1] + p) * vel[d]]
    F[1 + d] = F[1 + d] + p
    return F


def _jvp(eq, d, U, D):
    """f_d'(U) D."""
    if eq == "burgers":
        return [U[0] * D[0]]
    if eq == "buckley":
        return [8 * U[0] * (1 - U[0]) / (4 * U[0] ** 2 + (1 - U[0]) ** 2) ** 2 * D[0]]
    vel, p = _primitive(U)
    dvel = [(b - a * D[0]) / U[0] for a, b in zip(vel, D[1:-1])]
    dp = (GAMMA - 1) * (D[-1] - sum(a * b for a, b in zip(vel, D[1:-1]))
                        + 0.5 * sum(a * a for a in vel) * D[0])
    out = [D[1 + d]] + [D[1 + d] * a + U[1 + d] * b for a, b in zip(vel, dvel)]
    out[1 + d] = out[1 + d] + dp
    return out + [(D[-1] + dp) * vel[d] + (U[-1] + p) * dvel[d]]


def _speed(eq, d, U):
    if eq == "burgers":
        return U[0].abs()
    if eq == "buckley":  # at least the maximum over the admissible states [0, 1]
        u = 0.5
        for _ in range(60):  # 10u^3 - 15u^2 + 1 = 0, Newton from the inflection
            u -= (10 * u ** 3 - 15 * u ** 2 + 1) / (30 * u ** 2 - 30 * u)
        top = 8 * u * (1 - u) / (4 * u * u + (1 - u) ** 2) ** 2
        return _jvp(eq, d, U, [torch.ones_like(U[0])])[0].abs().clamp(min=top)
    vel, p = _primitive(U)
    return vel[d].abs() + (GAMMA * p / U[0]).sqrt()


def _eigen(d, vel, H):
    """(left rows, right columns) of the Euler flux Jacobian, each applied to
    a list of components."""
    q = 0.5 * sum(a * a for a in vel)
    c = ((GAMMA - 1) * (H - q)).sqrt()
    b1 = (GAMMA - 1) / (c * c)
    un = vel[d]

    def left(x):
        a = 0.5 * b1 * (q * x[0] - sum(v * y for v, y in zip(vel, x[1:-1])) + x[-1])
        b = 0.5 / c * (un * x[0] - x[1 + d])
        out = [a + b, x[0] - 2 * a, a - b]
        if len(vel) == 2:
            out.append(x[2 - d] - vel[1 - d] * x[0])
        return out

    def right(w):
        rest = w[3] if len(vel) == 2 else None
        total = w[0] + w[1] + w[2]
        out = [total] + [v * total for v in vel]
        out.append((H - un * c) * w[0] + q * w[1] + (H + un * c) * w[2])
        out[1 + d] = out[1 + d] + c * (w[2] - w[0])
        if rest is not None:
            out[2 - d] = out[2 - d] + rest
            out[3] = out[3] + vel[1 - d] * rest
        return out

    return left, right


def _enthalpy(U):
    vel, p = _primitive(U)
    return vel, (U[-1] + p) / U[0]


def _ghosts(eq, P, d, U, N, T, pos, t, h):
    """U, its derivative along the line N and across it T (or None) with two
    ghost points at each end; pos: the lines' other coordinate."""
    def sign(c):
        return -1.0 if eq == "burgers" or (eq == "euler" and c == 1 + d) else 1.0

    def end(a, c, side, which):
        kind = P["bc"][2 * d + side]
        if kind == "periodic":
            return a[:, -2:] if side == 0 else a[:, :2]
        if kind == "outflow":
            return (a[:, :1] if side == 0 else a[:, -1:]).expand(-1, 2)
        flip = (a[:, :2] if side == 0 else a[:, -2:]).flip(1)
        wall = flip * (sign(c) if which != "N" else -sign(c))
        if kind == "reflective":
            return wall
        fixed = torch.full_like(flip, P["inflow"][c] if which == "U" else 0.0)
        if kind == "dmr_bottom":
            return torch.where(pos[:, None] < P["dmr_x0"], fixed, wall)
        if kind == "dmr_top":
            n = a.shape[1]
            y = P["y0"] + (torch.arange(n, n + 2, dtype=torch.float64, device=a.device) + 0.5) * h
            xs = (P["dmr_x0"] + y / math.tan(P["dmr_angle"])
                  + P["dmr_speed"] * t / math.sin(P["dmr_angle"]))
            pre = torch.full_like(flip, P["pre"][c] if which == "U" else 0.0)
            return torch.where(pos[:, None] < xs[None], fixed, pre)
        return fixed

    def extend(F, which):
        return [torch.cat([end(a, c, 0, which), a, end(a, c, 1, which)], 1)
                for c, a in enumerate(F)]

    return extend(U, "U"), extend(N, "N"), None if T is None else extend(T, "T")


def _lines(eq, P, d, U, N, T, alpha, h, pos=None, t=0.0):
    """The terms of one direction: -d f-hat / h (for U), -d h-hat / h (for N),
    -d e-hat / h (for T, the central mixed flux) and the limited N."""
    n = U[0].shape[1]
    U, N, T = _ghosts(eq, P, d, U, N, T, pos, t, h)
    F, H = _flux(eq, d, U), _jvp(eq, d, U, N)
    at = lambda A, o: [a[:, o:o + n + 1] for a in A]  # noqa: E731  (interfaces, from point o - 2)
    fp = [0.5 * (f + alpha * u) for f, u in zip(F, U)]
    fm = [0.5 * (f - alpha * u) for f, u in zip(F, U)]
    hp = [0.5 * h * (g + alpha * v) for g, v in zip(H, N)]
    hm = [0.5 * h * (g - alpha * v) for g, v in zip(H, N)]
    stencil = [[at(A, o) for o in ((0, 1, 2) if up else (1, 2, 3))]
               for A, up in ((fp, 1), (hp, 1), (fm, 0), (hm, 0))]
    if eq == "euler":
        (velL, HL), (velR, HR) = _enthalpy(at(U, 1)), _enthalpy(at(U, 2))
        sL, sR = at(U, 1)[0].sqrt(), at(U, 2)[0].sqrt()
        roe = lambda a, b: (sL * a + sR * b) / (sL + sR)  # noqa: E731
        left, right = _eigen(d, [roe(a, b) for a, b in zip(velL, velR)], roe(HL, HR))
        chars = [[left(x) for x in s] for s in stencil]
    else:
        chars, right = stencil, lambda w: w
    fields = []
    for c in range(len(U)):
        p, hpl, m, hmi = ([x[c] for x in s] for s in chars)
        fields.append(_plus(p, hpl) + _plus(m[::-1], [-x for x in hmi[::-1]]))
    fhat = right(fields)
    hhat = []
    for c in range(len(U)):
        p, hpl, m, hmi = ([x[c] for x in s] for s in stencil)
        hhat.append((_derivative_plus(p, hpl)
                     - _derivative_plus(m[::-1], [-x for x in hmi[::-1]])) / h)
    back = lambda A: [-(a[:, 1:] - a[:, :-1]) / h for a in A]  # noqa: E731
    LU, LN, LT = back(fhat), back(hhat), None
    if T is not None:
        E = _jvp(eq, d, U, T)
        LT = back([(7 * (a[1] + a[2]) - a[0] - a[3]) / 12
                   for a in ([x[:, o:o + n + 1] for o in range(4)] for x in E)])
    mid = lambda A, o: [a[:, o:o + n] for a in A]  # noqa: E731
    if eq == "euler":
        left, right = _eigen(d, *_enthalpy(mid(U, 2)))
    else:
        left = right = lambda w: w
    us, vs = [left(mid(U, o)) for o in (1, 2, 3)], [left(mid(N, o)) for o in (1, 3)]
    lim = right([_limited([x[c] for x in us], [x[c] for x in vs], h) for c in range(len(U))])
    return LU, LN, LT, lim


def _operator(eq, P, fields, h, t):
    """(L^1, L^2 (, L^3)), (V~ (, W~)) and the wave speeds of a state: a list of
    fields, each a list of components [L][n] (1D) or [ny][nx]."""
    two = len(fields) == 3
    U, V = fields[:2]
    alpha = []
    for d in range(2 if two else 1):
        s = _speed(eq, d, [a.detach() for a in U])
        alpha.append(s.max() if two else s.max(1, keepdim=True).values)
    if not two:
        LU, LV, _, Vt = _lines(eq, P, 0, U, V, None, alpha[0], h[0])
        return [LU, LV], [Vt], alpha
    ny, nx = U[0].shape
    x = _centers(P["x0"], P["x1"], nx).to(U[0].device)
    y = _centers(P["y0"], P["y1"], ny).to(U[0].device)
    W = fields[2]
    tr = lambda A: [a.t() for a in A]  # noqa: E731
    LU, LV, LW, Vt = _lines(eq, P, 0, U, V, W, alpha[0], h[0], y, t)
    MU, MW, MV, Wt = (tr(A) for A in _lines(eq, P, 1, tr(U), tr(W), tr(V), alpha[1], h[1], x, t))
    add = lambda A, B: [a + b for a, b in zip(A, B)]  # noqa: E731
    return [add(LU, MU), add(LV, MV), add(LW, MW)], [Vt, Wt], alpha


def _step(eq, P, fields, h, t, t_end):
    """One SSP-RK3 step; t: float (2D) or [L][1]. Returns the fields and t."""
    two = len(fields) == 3

    def stage(x, time):
        L, lim, alpha = _operator(eq, P, x, h, time)
        return [[b + dt * a for a, b in zip(A, B)] for A, B in zip(L, [x[0]] + lim)]

    L, lim, alpha = _operator(eq, P, fields, h, t)
    rate = sum(a / b for a, b in zip(alpha, h))
    dt = CFL / rate
    lands = dt >= t_end - t
    dt = torch.where(lands, t_end - t, dt)
    base = [fields[0]] + lim
    one = [[b + dt * a for a, b in zip(A, B)] for A, B in zip(L, base)]
    mix = lambda c, A, B: [[c * x + (1 - c) * y for x, y in zip(a, b)] for a, b in zip(A, B)]  # noqa: E731
    second = mix(0.75, base, stage(one, t + dt))
    third = mix(1 / 3, base, stage(second, t + 0.5 * dt))
    tn = torch.where(lands, torch.full_like(t, t_end), t + dt)
    if not two:  # finished instances stay
        live = t < t_end
        third = [[torch.where(live, a, b) for a, b in zip(A, B)] for A, B in zip(third, fields)]
        tn = torch.where(live, tn, t)
    return third, tn


def _advance(case, P, x, h, t):
    eq = EQUATION[case["problem"]]
    if case["call"] == "gradient":
        for _ in range(2 * case["steps"]):
            x, t = _step(eq, P, x, h, t, _gradient_end(case))
    else:
        for _ in range(case["steps"]):
            x, t = _step(eq, P, x, h, t, 1e30)
    return x, t


def _exact_group(case, P, fields, lam, h):
    """Outputs of one group of lines: fields (and cotangents) as [L][m][n]
    (1D) or [1][m][ny][nx]; by name, each in that shape."""
    eq, two = EQUATION[case["problem"]], case["nx"] != 0
    split = lambda a: list(a[0]) if two else [a[:, c] for c in range(a.shape[1])]  # noqa: E731
    join = lambda A: torch.stack(A)[None] if two else torch.stack(A, 1)  # noqa: E731
    t = torch.zeros((), dtype=torch.float64, device="cuda")
    if not two:
        t = t.expand(fields[0].shape[0], 1).clone()
    if case["call"] == "rhs":
        L, lim, _ = _operator(eq, P, [split(a) for a in fields], h, t)
        names = ("L1", "L2", "L3"), ("Vt", "Wt")
        return {**dict(zip(names[0], map(join, L))), **dict(zip(names[1], map(join, lim)))}
    if lam is not None:
        fields = [a.detach().clone().requires_grad_(True) for a in fields]
    x, t = _advance(case, P, [split(a) for a in fields], h, t)
    x = [join(a) for a in x]
    out = dict(zip("UVW", (a.detach() for a in x)))
    if case["call"] != "gradient":
        out["t"] = t.reshape(-1)
    if lam is not None:
        g = torch.autograd.grad(x, fields, lam)
        out.update(zip(("gU", "gV", "gW"), g))
    return out


def exact(case, seed):
    P = _grid(case)
    fields = [a.double() for a in _fields(case, seed)]
    lam = _cotangents(case, seed, fields) if case["call"] in ("adjoint", "gradient") else None
    eq = EQUATION[case["problem"]]
    if case["nx"] != 0:
        shape = (1, 4 if eq == "euler" else 1, case["ny"], case["nx"])
        h = [(P["x1"] - P["x0"]) / case["nx"], (P["y1"] - P["y0"]) / case["ny"]]
        with torch.set_grad_enabled(lam is not None):
            out = _exact_group(case, P, [a.reshape(shape) for a in fields],
                               lam and [a.reshape(shape) for a in lam], h)
        return {k: a.reshape(-1) for k, a in out.items()}
    nx, m = _sizes(case), 3 if eq == "euler" else 1
    rows = {}
    parts = [a.split([m * n for n in nx]) for a in fields + (lam or [])]
    for n in sorted(set(nx)):
        who = [k for k, size in enumerate(nx) if size == n]
        group = [torch.stack([a[k] for k in who]).reshape(-1, m, n) for a in parts]
        with torch.set_grad_enabled(lam is not None):
            out = _exact_group(case, P, group[:2], group[2:] or None, [(P["x1"] - P["x0"]) / n])
        for name, a in out.items():
            a = a.reshape(len(who), -1)
            for j, k in enumerate(who):
                rows.setdefault(name, {})[k] = a[j]
    return {name: torch.cat([r[k] for k in range(len(nx))]) for name, r in rows.items()}
