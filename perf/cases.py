"""What a user of the library has it do, as measurable cases.

Every single-problem case is one solve through the public binding: write the
initial state into the problem, advance it with the library's default launch
and width, read the final state (all on the device).  The batched cases advance
a mixed set of problems in one call; the served case submits host requests and
waits for their results.  Sizes are those of the configurations, tests and
benchmark of this repository (N from 2^10 to 2^21 and any integer between) and
ragged neighbours of them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1705_03162_gb300 import inputs as I
from paper_1705_03162_gb300 import swept as S

# flops of one point-update (an FMA is two): heat one stencil, KS and Euler two
# Runge-Kutta stages
_FLOPS = {"heat": 5.0, "ks": 22.0, "euler": 142.0}


def listed():
    return [
        # the smallest call: a few steps of a small grid between two actions of
        # the caller (a coupled model, a control loop); launch latency counts
        dict(name="heat_f64_short_call", kind="solve", eq="heat", bc="periodic", dtype="f64", n=1024, steps=64),
        # the heat configuration: N = 1024, r = 0.25, 4096 steps
        dict(name="heat_f64_1024", kind="solve", eq="heat", bc="periodic", dtype="f64", n=1024, steps=4096),
        # a KS study on a mid-size grid whose N is no multiple of anything
        dict(name="ks_f64_10007", kind="solve", eq="ks", bc="periodic", dtype="f64", n=10007, steps=2000),
        # the paper's insulated-end heat problem on a ragged mid-size grid
        dict(name="heat_f64_reflective_50001", kind="solve", eq="heat", bc="reflective", dtype="f64", n=50001,
             steps=2000),
        # the headline problem's grid, a tenth of its 10^4 steps
        dict(name="ks_f64_2e20", kind="solve", eq="ks", bc="periodic", dtype="f64", n=1 << 20, steps=1000),
        # single precision where it is accurate enough: heat, mid-size
        dict(name="heat_f32_2e17", kind="solve", eq="heat", bc="periodic", dtype="f32", n=1 << 17, steps=4000),
        # single-precision KS beyond the paper's largest grid, ragged
        dict(name="ks_f32_2000003", kind="solve", eq="ks", bc="periodic", dtype="f32", n=2000003, steps=1000),
        # Sod tube to t = 0.2 (N steps at dt / dx = 0.2)
        dict(name="sod_f64_4096", kind="solve", eq="euler", bc="dirichlet", dtype="f64", n=4096, steps=4096),
        # a smooth flow on a large periodic grid: limited reconstruction everywhere
        dict(name="euler_f64_periodic_200000", kind="solve", eq="euler", bc="periodic", dtype="f64", n=200000,
             steps=200),
        # an ensemble of mixed heat and KS problems in one batched advance
        dict(name="batch_f64", kind="batch", dtype="f64", count=256, n_max=1 << 16, steps_lo=400, steps_hi=1600,
             set_seed=1),
        # the same in single precision, longer
        dict(name="batch_f32", kind="batch", dtype="f32", count=256, n_max=1 << 16, steps_lo=2000, steps_hi=10000,
             set_seed=2),
        # a burst of mixed requests to the server, host buffers in and out
        dict(name="serve_f64", kind="serve", dtype="f64", count=24, n_max=1 << 17, steps_lo=100, steps_hi=1000,
             set_seed=3),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["batch", "batch", "serve"])
    if kind == "solve":
        eq, bc, dtype = rng.choice([("heat", "periodic", "f64"), ("heat", "reflective", "f64"),
                                    ("ks", "periodic", "f64"), ("ks", "periodic", "f64"),
                                    ("heat", "periodic", "f32"), ("heat", "reflective", "f32"),
                                    ("ks", "periodic", "f32"), ("euler", "dirichlet", "f64"),
                                    ("euler", "periodic", "f64")])
        top = 1 << 21 if dtype == "f32" else (200000 if eq == "euler" else 1 << 20)
        n = _log_uniform(rng, 1000, top)
        n = rng.choice([n, n | 1, max(1024, n // 32 * 32), 1 << (n.bit_length() - 1)])
        n = max(n, 1000)
        # at most the work of the largest listed case of the equation and type
        most = {("heat", "f64"): 1.0e9, ("ks", "f64"): 1.0e9, ("heat", "f32"): 2.0e9, ("ks", "f32"): 2.0e9,
                ("euler", "f64"): 1.6e7}[(eq, dtype)]
        steps = _log_uniform(rng, 32, 4096)
        steps = max(1, min(steps, int(most / n)))
        return dict(kind="solve", eq=eq, bc=bc, dtype=dtype, n=n, steps=steps)
    if kind == "batch":
        dtype = rng.choice(["f64", "f32"])
        lo, hi = (400, 1600) if dtype == "f64" else (2000, 10000)
        return dict(kind="batch", dtype=dtype, count=_log_uniform(rng, 32, 192), n_max=rng.choice([1 << 14, 1 << 16]),
                    steps_lo=lo, steps_hi=hi, set_seed=rng.randrange(1 << 20))
    return dict(kind="serve", dtype="f64", count=rng.randrange(6, 25), n_max=rng.choice([1 << 14, 1 << 17]),
                steps_lo=100, steps_hi=1000, set_seed=rng.randrange(1 << 20))


def _seeded_state(eq, bc, n, seed):
    """(spec, FP64 initial state of shape (nv, N)): each equation's initial
    condition, its free parts drawn from the seed."""
    g = np.random.default_rng([seed, n, {"heat": 0, "ks": 1, "euler": 2}[eq]])
    if eq == "heat":
        # the configuration's low modes with drawn amplitudes (cosines keep
        # insulated ends insulated)
        spec = I.heat_spec(n, bc=bc)
        f, span = (np.sin, n) if bc == "periodic" else (np.cos, 2.0 * (n - 1))
        x = 2.0 * math.pi * np.arange(n) / span
        u = f(x)
        for k in range(2, 10):
            u += g.uniform(-0.1, 0.1) * f(k * x)
        return spec, u[None, :]
    if eq == "ks":
        spec = I.ks_spec(n)
        return spec, (I.ks_ic(n, spec.dx) + 0.05 * g.uniform(-1.0, 1.0, n))[None, :]
    if bc == "dirichlet":
        # Sod's states, a few per cent of them drawn
        left = (1.0 + 0.05 * g.uniform(), 0.0, 1.0 + 0.05 * g.uniform())
        right = (0.125 + 0.01 * g.uniform(), 0.0, 0.1 + 0.01 * g.uniform())
        dx = 1.0 / n
        spec = I.ProblemSpec("euler", "dirichlet", n, dx, 0.2 * dx, left=left, right=right)
        return spec, I.sod_ic(n, spec.gamma, left, right)
    spec = I.sod_spec(n, bc="periodic")
    x = (np.arange(n) + 0.5) / n
    p0, p1 = g.uniform(0.0, 2.0 * math.pi, 2)
    rho = 1.0 + 0.3 * np.sin(2 * math.pi * x + p0) + 0.02 * g.uniform(-1.0, 1.0, n)
    vel = 0.4 * np.cos(2 * math.pi * x + p1)
    p = 1.0 + 0.2 * np.cos(4 * math.pi * x + p0)
    return spec, np.stack([rho, rho * vel, p / (spec.gamma - 1.0) + 0.5 * rho * vel * vel])


def _members(case):
    """(eq, bc, N, steps) of a mixed set: sizes log-uniform on [2^10, n_max] as
    any integer, steps uniform (fixed by set_seed, not by the input seed)."""
    g = np.random.default_rng(case["set_seed"])
    kinds = ([("heat", "periodic"), ("ks", "periodic")] if case["kind"] == "batch" else
             [("heat", "periodic"), ("ks", "periodic"), ("euler", "dirichlet")])
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(g.uniform(math.log(1 << 10), math.log(case["n_max"])))))
        out.append((*kinds[i % len(kinds)], n, int(g.integers(case["steps_lo"], case["steps_hi"] + 1))))
    return out


def _np_dtype(case):
    return np.float64 if case["dtype"] == "f64" else np.float32


def prepare(case, seed):
    dt = _np_dtype(case)
    if case["kind"] == "solve":
        spec, u = _seeded_state(case["eq"], case["bc"], case["n"], seed)
        u0 = torch.from_numpy(np.ascontiguousarray(u.astype(dt))).cuda()
        return dict(case=case, problem=S.Problem(spec, u0, case["dtype"]), u0=u0, out=torch.empty_like(u0))
    members = _members(case)
    states = [_seeded_state(eq, bc, n, seed + 1000 * i) for i, (eq, bc, n, _) in enumerate(members)]
    steps = [m[3] for m in members]
    if case["kind"] == "serve":
        # the server lives across bursts, as a service's would
        return dict(case=case, server=S.Server(round_target_ms=20.0), specs=[s for s, _ in states],
                    u0=[np.ascontiguousarray(u.astype(dt)) for _, u in states], steps=steps)
    flat = torch.from_numpy(np.concatenate([u.astype(dt).ravel() for _, u in states])).cuda()
    out = torch.empty_like(flat)
    sizes = [u.size for _, u in states]
    u0s, outs = flat.split(sizes), out.split(sizes)
    problems = [S.Problem(spec, u, case["dtype"]) for (spec, _), u in zip(states, u0s)]
    # node widths of about 2048 points fitted to each N, the choice tune_width
    # makes for such a set
    widths = [S.fit_width(spec.eq, spec.n_points, 2048) for spec, _ in states]
    return dict(case=case, batch=S.Batch(), problems=problems, u0=u0s, outs=outs, out=out, steps=steps, widths=widths)


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        p = state["problem"]
        p.write(state["u0"])
        p.advance(case["steps"], "swept")
        return p.read(state["out"])
    if case["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(spec, u, st) for spec, u, st in zip(state["specs"], state["u0"], state["steps"])]
        return [srv.wait(i)[0] for i in ids]
    for p, u in zip(state["problems"], state["u0"]):
        p.write(u)
    state["batch"].advance_ex(state["problems"], state["steps"], ["swept"] * len(state["problems"]),
                              state["widths"], launch="graph")
    for p, o in zip(state["problems"], state["outs"]):
        p.read(o)
    return state["out"]


def work(case):
    size = 8 if case["dtype"] == "f64" else 4
    members = ([(case["eq"], case["bc"], case["n"], case["steps"])] if case["kind"] == "solve" else _members(case))
    # the initial state read once, the final state written once
    return {"bytes": float(sum(2 * size * n * (3 if eq == "euler" else 1) for eq, _, n, _ in members)),
            "flops": float(sum(_FLOPS[eq] * n * st for eq, _, n, st in members))}


# ---------------------------------------------------------------------------
# The same solves in 64 bits with plain torch operations.
# ---------------------------------------------------------------------------
def _exact_heat(spec, u, steps):
    fo = spec.alpha * spec.dt / (spec.dx * spec.dx)
    periodic = spec.bc == "periodic"
    for _ in range(steps):
        if periodic:
            lo, hi = torch.roll(u, 1), torch.roll(u, -1)
        else:
            lo, hi = torch.cat([u[1:2], u[:-1]]), torch.cat([u[1:], u[-2:-1]])
        u = u + fo * (lo + hi - 2.0 * u)
    return u


def _exact_ks(spec, u, steps):
    dx2 = spec.dx * spec.dx

    def f(v):
        m2, m1, p1, p2 = (torch.roll(v, s) for s in (2, 1, -1, -2))
        return -((p1 * p1 - m1 * m1) / (4.0 * spec.dx) + (p1 - 2.0 * v + m1) / dx2 +
                 (p2 - 4.0 * p1 + 6.0 * v - 4.0 * m1 + m2) / (dx2 * dx2))

    for _ in range(steps):
        u = u + spec.dt * f(u + 0.5 * spec.dt * f(u))
    return u


def _exact_euler(spec, q, steps):
    gam = spec.gamma
    lam = spec.dt / spec.dx
    ends = []
    for r, v, p in (spec.left, spec.right):
        s = torch.tensor([r, r * v, p / (gam - 1.0) + 0.5 * r * v * v], dtype=torch.float64, device=q.device)
        ends.append(s[:, None].expand(3, 2))

    def primitive(s):
        v = s[1] / s[0]
        return v, (gam - 1.0) * (s[2] - 0.5 * s[1] * v)

    def rate(s):
        # two ghost cells each side, interfaces between padded cells 1|2 .. N+1|N+2
        g = (torch.cat([s[:, -2:], s, s[:, :2]], 1) if spec.bc == "periodic" else
             torch.cat([ends[0], s, ends[1]], 1))
        p = primitive(g)[1]
        d = p[1:] - p[:-1]
        dm, dc, dp = d[:-2], d[1:-1], d[2:]
        a, b = g[:, 1:-2], g[:, 2:-1]
        one, zero = torch.ones_like(dc), torch.zeros_like(dc)
        same_l, same_r = dc.sign() * dm.sign() > 0, dp.sign() * dc.sign() > 0
        hl = torch.where(same_l, 0.5 * torch.minimum(dc / torch.where(same_l, dm, one), one), zero)
        hr = torch.where(same_r, 0.5 * torch.minimum(dc / torch.where(same_r, dp, one), one), zero)
        ql, qr = a + hl * (b - a), b + hr * (a - b)

        def flux(s):
            v, p = primitive(s)
            return torch.stack([s[1], s[1] * v + p, v * (s[2] + p)])

        wl, wr = ql[0].sqrt(), qr[0].sqrt()
        vs = (wl * ql[1] / ql[0] + wr * qr[1] / qr[0]) / (wl + wr)
        es = (wl * ql[2] / ql[0] + wr * qr[2] / qr[0]) / (wl + wr)
        speed = (gam * (gam - 1.0) * (es - 0.5 * vs * vs)).sqrt() + vs.abs()
        fx = 0.5 * (flux(ql) + flux(qr) + speed * (ql - qr))
        return fx[:, 1:] - fx[:, :-1]

    for _ in range(steps):
        q = q - lam * rate(q - 0.5 * lam * rate(q))
    return q


def _exact_one(spec, u, steps):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = torch.from_numpy(np.ascontiguousarray(u.astype(np.float64))).to(dev)
    if spec.eq == "heat":
        return _exact_heat(spec, t[0], steps)[None, :]
    if spec.eq == "ks":
        return _exact_ks(spec, t[0], steps)[None, :]
    return _exact_euler(spec, t, steps)


def exact(case, seed):
    dt = _np_dtype(case)
    if case["kind"] == "solve":
        spec, u = _seeded_state(case["eq"], case["bc"], case["n"], seed)
        return _exact_one(spec, u.astype(dt), case["steps"])
    members = _members(case)
    if case["kind"] == "batch":
        # hundreds of long solves in small torch operations take minutes
        return None
    out = []
    for i, (eq, bc, n, st) in enumerate(members):
        spec, u = _seeded_state(eq, bc, n, seed + 1000 * i)
        # the Euler members' many small operations would pass the time limit
        out.append(None if eq == "euler" else _exact_one(spec, u.astype(dt), st))
    return out
