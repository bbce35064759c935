"""The performance cases: what a program that uses this library has it do, through its public entry points.

One pass is a whole call as such a program makes it: initial data on the host in, the adaptive solve on the GPU, the
solution on the host out.  Three kinds:

- "solve": one `Solver`, kept by the program and given new data with reset() (or made anew for each solve, "fresh"),
  stepped to its end time, read with leaves() or uniform();
- "batch": independent reaction-diffusion problems of uneven size advanced together by a `Batch`;
- "serve": a mixed stream of requests through a `Server`, all submitted at once and served until none is left.

Sizes and parameters are those of the repository's workloads: the 1D Burgers problem at L = 10, the 2D Euler
quadrant problem at L = 10, the paper's 2D Burgers and AUSM+ Euler problems, the 3D blast at L = 7 and 8, the
reaction-diffusion batch with L = 7..10, the serving mix with 1D L = 10..14, and the finite-volume reference solve on
the full grid.  `iters` is the nominal number of fine iterations; the end time is that many steps at the problem's
nominal wave speed.
"""
import functools
import math
import random

import numpy as np

import paper_1905_08717_gb300 as mr
from paper_1905_08717_gb300 import inputs

_DIM = {"advection1d": 1, "burgers1d": 1, "euler2d": 2, "burgers2d": 2, "rd2d": 2, "blast3d": 3}
_VARS = {"advection1d": 1, "burgers1d": 1, "euler2d": 4, "burgers2d": 1, "rd2d": 1, "blast3d": 5}


def _solve(problem, L, iters, **kw):
    case = {"kind": "solve", "problem": problem, "L": L, "min_level": 3, "eps": 1e-3, "rk": 3, "time": "lt",
            "precision": "fp64", "adapt": "every", "flux": "default", "iters": iters, "fresh": False,
            "read": "leaves"}
    case.update(kw)
    return case


def listed():
    return [
        # a small one-dimensional solve made from nothing: creation, two macro steps, result (latency and launches)
        dict(_solve("burgers1d", 10, 512, min_level=2, fresh=True), name="burgers1d_L10"),
        # the smallest call: one macro step of local time stepping on the fixed two-level tree of the convergence study
        dict(_solve("advection1d", 9, 8, min_level=6, eps=0.0, adapt="never"), name="advection1d_L9_two_level"),
        # the headline: the whole 2D Euler quadrant solve with local time stepping
        dict(_solve("euler2d", 10, 1920), name="euler2d_L10"),
        # its opening in mixed precision, read back on the finest grid
        dict(_solve("euler2d", 10, 384, precision="mixed", read="uniform"), name="euler2d_L10_mixed"),
        # the same method with one global time step, a size smaller
        dict(_solve("euler2d", 9, 192, time="gts"), name="euler2d_L9_gts"),
        # the paper's Euler experiment: AUSM+, RK2, a coarser threshold
        dict(_solve("euler2d", 10, 768, rk=2, flux="ausm", eps=1e-2), name="euler2d_L10_ausm_rk2"),
        # the paper's 2D Burgers experiment: RK2, zero walls
        dict(_solve("burgers2d", 10, 1536, rk=2), name="burgers2d_L10_rk2"),
        # the 3D blast in double precision
        dict(_solve("blast3d", 7, 48), name="blast3d_L7"),
        # the largest state: the 3D blast on 256^3 in mixed precision
        dict(_solve("blast3d", 8, 32, precision="mixed"), name="blast3d_L8_mixed"),
        # a batch of uneven reaction-diffusion problems
        {"kind": "batch", "count": 24, "L_lo": 7, "L_hi": 10, "rk": 2, "t_end": 0.02, "name": "rd2d_batch_24"},
        # a server with a mixed load: 1D Burgers, 2D reaction-diffusion, 3D blast, in mixed precision
        {"kind": "serve", "count": 12, "L3_hi": 7, "name": "serve_12"},
        # the finite-volume reference: every cell of the finest grid, one global step
        dict(_solve("euler2d", 9, 8, min_level=7, eps=0.0, time="gts", adapt="never", read="uniform"),
             name="euler2d_L9_fv"),
    ]


def draw(rng):
    u = rng.random()
    if u < 0.08:
        lo = rng.randint(6, 8)
        return {"kind": "batch", "count": rng.randint(2, 23), "L_lo": lo, "L_hi": rng.randint(lo, 10),
                "rk": rng.choice((2, 3)), "t_end": round(10.0 ** rng.uniform(-2.6, -1.7), 5)}
    if u < 0.16:
        return {"kind": "serve", "count": rng.randint(2, 15), "L3_hi": rng.randint(5, 7)}
    if u < 0.28:  # the full grid
        problem, lo, hi = rng.choice((("burgers1d", 6, 14), ("burgers2d", 6, 9), ("euler2d", 6, 9)))
        L = rng.randint(lo, hi)
        return _solve(problem, L, rng.randint(3, 11), min_level=L - rng.randint(0, 2), eps=0.0, rk=rng.choice((2, 3)),
                      time="gts", adapt="never", read=rng.choice(("leaves", "uniform")))
    problem, lo, hi, most = rng.choice((("advection1d", 6, 12, 512), ("burgers1d", 7, 14, 512), ("euler2d", 6, 10, 512),
                                        ("euler2d", 6, 10, 512), ("burgers2d", 6, 10, 512), ("rd2d", 6, 10, 256),
                                        ("blast3d", 4, 7, 48)))
    L = rng.randint(lo, hi)
    if problem == "advection1d":
        return _solve(problem, L, rng.randint(5, 96), min_level=L - rng.randint(2, 4), eps=0.0, adapt="never",
                      rk=rng.choice((2, 3)), time=rng.choice(("lt", "gts")))
    return _solve(problem, L, int(8 * (most / 8) ** rng.random()), min_level=max(rng.randint(2, 4), L - 7),
                  eps=round(10.0 ** rng.uniform(-4.0, -2.0), 6), rk=rng.choice((2, 3)),
                  time=rng.choice(("lt", "lt", "gts")), precision=rng.choice(("fp64", "fp64", "mixed")),
                  adapt=rng.choice(("every", "every", "macro")),
                  flux=rng.choice(("default", "ausm")) if problem in ("euler2d", "blast3d") else "default",
                  fresh=rng.random() < 0.2, read=rng.choice(("leaves", "leaves", "uniform")))


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=2)
def _ball(L):
    """The blast's geometry on the finest grid: the share of each cell inside the ball of radius 0.1."""
    n = 1 << L
    c2 = (((np.arange(n) + 0.5) / n - 0.5) ** 2).astype(np.float64)
    r = np.sqrt(c2[None, None, :] + c2[None, :, None] + c2[:, None, None])
    return np.clip((0.1 - r) * n + 0.5, 0.0, 1.0)


def _data(problem, L, rng, **kw):
    """The repository's problem and its finest-level cell averages, varied by the seed."""
    if problem == "advection1d":
        p, q = inputs.advection_gaussian_1d(L=L, **kw)
        q = rng.uniform(0.8, 1.2) * q
    elif problem == "burgers1d":
        p, q = inputs.burgers_1d(L=L, **kw)
        q = rng.uniform(0.9, 1.1) * np.roll(q, rng.randrange(1 << L), axis=1)
    elif problem == "euler2d":
        p, q = inputs.euler_2d_quadrants(L=L, seed=1 + rng.randrange(1 << 20), **kw)
    elif problem == "burgers2d":
        p, q = inputs.burgers_2d_paper(L=L, **kw)
        q = rng.uniform(0.9, 1.1) * q
    elif problem == "rd2d":
        p, q = inputs.rd_bumps_2d(L=L, seed=rng.randrange(1 << 20), midpoint=True, **kw)
    else:
        p, q = inputs.euler_3d_blast(L=3, **kw)  # the parameters; the data below
        p = p.replace(max_level=L, name="euler3d_blast_L%d" % L)
        q = np.zeros((5,) + (1 << L,) * 3)
        q[0] = 1.0
        q[4] = (1.0 + (rng.uniform(8.0, 12.0) - 1.0) * _ball(L)) / (p.phys[0] - 1.0)
    return p, np.ascontiguousarray(q)


def _dt(problem, L):
    """The fine step at the problem's nominal wave speed (CFL 0.5)."""
    dx = 0.5 ** L
    if problem == "rd2d":
        return 0.5 * dx * dx / (4.0 * 1e-3)
    return 0.5 * dx / {"advection1d": 1.0, "burgers1d": 1.0, "euler2d": 3.75, "burgers2d": 2.0, "blast3d": 11.2}[problem]


def _make(case, rng):
    kw = dict(min_level=case["min_level"], eps=case["eps"], rk_order=case["rk"])
    if case["problem"] == "advection1d":
        kw = dict(rk_order=case["rk"])
    if case["problem"] == "burgers1d":
        kw["eps"] = case["eps"] or 1e-3
    p, q = _data(case["problem"], case["L"], rng, **kw)
    p = p.replace(min_level=case["min_level"], eps=case["eps"],
                  time_mode=inputs.TIME_GTS if case["time"] == "gts" else inputs.TIME_LT,
                  adapt_mode={"never": inputs.ADAPT_NEVER, "macro": inputs.ADAPT_MACRO,
                              "every": inputs.ADAPT_EVERY}[case["adapt"]],
                  precision=inputs.PREC_MIXED if case["precision"] == "mixed" else inputs.PREC_FP64,
                  flux=inputs.FLUX_AUSM_PLUS if case["flux"] == "ausm" else inputs.FLUX_DEFAULT)
    return p, q, case["iters"] * _dt(case["problem"], case["L"])


def _requests(case, rng):
    out = []
    for i in range(case["count"]):
        eps = 10.0 ** rng.uniform(-4.0, -2.0)
        kind = ("burgers1d", "rd2d", "blast3d")[i % 3]
        if kind == "burgers1d":
            L, its = 10 + i // 3 % 5, rng.randint(32, 128)
            p, q = _data(kind, L, rng, eps=eps, min_level=L - 7)
        elif kind == "rd2d":
            L, its = 8 + i // 3 % 3, rng.randint(16, 64)
            p, q = _data(kind, L, rng, eps=eps)
        else:
            L, its = max(case["L3_hi"] - i // 3 % 3, 4), rng.randint(8, 24)
            p, q = _data(kind, L, rng, eps=eps, min_level=max(L - 4, 2))
        out.append((p.replace(precision=inputs.PREC_MIXED), q, its * _dt(kind, L)))
    return out


def _room(p, read="leaves"):
    """The program's own arrays for the leaves, for the largest tree that it allows; the mixed mode stores its values
    in 32 bits, and they are kept as such.  None: it reads the finest grid."""
    if read == "uniform":
        return None
    n = min(1 << (p.dim * p.max_level), 1 << 20)
    return (np.zeros((n, 4), np.int32),
            np.zeros((n, p.nvars()), np.float32 if p.precision == inputs.PREC_MIXED else np.float64))


def prepare(case, seed):
    rng = random.Random(seed)
    if case["kind"] == "batch":
        probs, qs = [], []
        for i in range(case["count"]):
            L = case["L_lo"] + i % (case["L_hi"] - case["L_lo"] + 1)
            p, q = _data("rd2d", L, rng, eps=rng.choice((1e-3, 1e-4)), rk_order=case["rk"])
            probs.append(p)
            qs.append(q)
        return {"case": case, "problems": probs, "q": qs, "room": [_room(p) for p in probs]}
    if case["kind"] == "serve":
        requests = _requests(case, rng)
        return {"case": case, "requests": requests, "room": [_room(p) for p, _, _ in requests]}
    p, q, t_end = _make(case, rng)
    state = {"case": case, "p": p, "q": q, "t_end": t_end, "room": _room(p, case["read"])}
    if case["problem"] == "advection1d":
        state["tree"] = inputs.two_level_map_1d(case["L"])
    if not case["fresh"]:
        state["solver"] = mr.Solver(p, q)
    return state


# ------------------------------------------------------------------ one pass
def _result(solver, room):
    """What a program reads at the end: the finest grid, or the leaves into its own arrays."""
    if room is None:
        t = np.float32 if solver.p.precision == inputs.PREC_MIXED else np.float64
        return solver.uniform().astype(t, copy=False)
    keys, values = solver.leaves()
    room[0][: len(keys)] = keys
    room[1][: len(keys)] = values
    return room


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = mr.Batch(state["problems"], state["q"])
        batch.step(case["t_end"])
        out = [_result(s, r) for s, r in zip(batch.instances, state["room"])]
        batch.close()
        return out
    if case["kind"] == "serve":
        server = mr.Server(64 << 30, 96)
        ids = [server.submit(p, q, t) for p, q, t in state["requests"]]
        left = len(ids)
        while left:
            server.advance()
            left -= len(server.poll())
        out = [_result(server.result(i), r) for i, r in zip(ids, state["room"])]
        server.close()
        return out
    if case["fresh"]:
        solver = mr.Solver(state["p"], state["q"])
    else:
        solver = state["solver"]
        solver.reset(state["q"])
    if "tree" in state:
        solver.set_tree(state["tree"])
    solver.step(state["t_end"])
    out = _result(solver, state["room"])
    if case["fresh"]:
        solver.close()
    return out


# ------------------------------------------------------------------ the work of one pass
#: operations of one leaf in one stage, counting each face flux once
_FLOPS = {"advection1d": 12, "burgers1d": 30, "burgers2d": 55, "rd2d": 25, "euler2d": 260, "blast3d": 480}
#: leaves that one fine iteration advances with local time stepping, in units of 2^{(d-1) L} (fronts of codimension one)
_FRONT = {"burgers1d": 30.0, "burgers2d": 30.0, "rd2d": 40.0, "euler2d": 35.0, "blast3d": 8.0}


def _work_solve(problem, L, iters, rk, full, gts, read):
    d, m = _DIM[problem], _VARS[problem]
    cells = 2.0 ** (d * L)
    leaves = cells if full else min(cells, _FRONT[problem] * 2.0 ** ((d - 1) * L))
    updates = leaves * iters * (2.0 if gts and not full else 1.0)
    out = 8.0 * m * cells if read == "uniform" else (8.0 * m + 16.0) * leaves
    return 8.0 * m * cells + out, updates * rk * _FLOPS[problem]


def work(case):
    """Bytes: the initial data read once and the result written once (a solve's state can stay on the chip between).
    Operations: those of the leaves' stages, with the leaves of an adaptive solve taken as fronts of codimension one."""
    if case["kind"] == "solve":
        b, f = _work_solve(case["problem"], case["L"], case["iters"], case["rk"],
                           case["adapt"] == "never", case["time"] == "gts", case["read"])
    elif case["kind"] == "batch":
        b = f = 0.0
        levels = range(case["L_lo"], case["L_hi"] + 1)
        for L in levels:
            x = _work_solve("rd2d", L, max(1.0, case["t_end"] / _dt("rd2d", L)), case["rk"], False, False, "leaves")
            b, f = b + x[0] * case["count"] / len(levels), f + x[1] * case["count"] / len(levels)
    else:
        b = f = 0.0
        for i in range(case["count"]):
            kind, L, its, rk = (("burgers1d", 12, 80, 3), ("rd2d", 9, 40, 2), ("blast3d", case["L3_hi"] - 0.7, 16, 3))[i % 3]
            x = _work_solve(kind, L, its, rk, False, False, "leaves")
            b, f = b + x[0], f + x[1]
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the exact result on the full grid
def _minmod(a, b):
    return np.where(a * b <= 0.0, 0.0, np.where(np.abs(a) < np.abs(b), a, b))


def _speed(p, q):
    if p.equation == inputs.EQ_BURGERS:
        return p.dim * np.abs(q[0]).max()
    pr = (p.phys[0] - 1.0) * (q[-1] - 0.5 * (q[1:-1] ** 2).sum(axis=0) / q[0])
    c = np.sqrt(p.phys[0] * pr / q[0])
    return (np.abs(q[1:-1] / q[0]).sum(axis=0) + p.dim * c).max()


def _rhs(p, q):
    """-div F by the second-order finite volumes of the full grid: limited slopes, Godunov (Burgers) or HLL (Euler)."""
    gam, h, out = p.phys[0], 0.5 ** p.max_level, np.zeros_like(q)
    w = q.copy()
    if p.equation == inputs.EQ_EULER:
        w[1:-1] = q[1:-1] / q[0]
        w[-1] = (gam - 1.0) * (q[-1] - 0.5 * (q[1:-1] * w[1:-1]).sum(axis=0))
    for k in range(p.dim):
        ax = q.ndim - 1 - k
        pad = [(0, 0)] * q.ndim
        pad[ax] = (2, 2)
        if p.bc[k] == inputs.BC_DIRICHLET0:  # odd mirror
            g = np.pad(w, pad, mode="symmetric")
            e = np.moveaxis(g, ax, -1)
            e[..., :2] *= -1.0
            e[..., -2:] *= -1.0
        else:
            g = np.pad(w, pad, mode="wrap" if p.bc[k] == inputs.BC_PERIODIC else "symmetric")
        g = np.moveaxis(g, ax, -1)
        s = np.diff(g, axis=-1)
        half = 0.5 * _minmod(s[..., :-1], s[..., 1:])
        left, right = g[..., 1:-2] + half[..., :-1], g[..., 2:-1] - half[..., 1:]
        if p.equation == inputs.EQ_BURGERS:
            fl, fr = 0.5 * left * left, 0.5 * right * right
            f = np.where(left <= right, np.where(left > 0.0, fl, np.where(right < 0.0, fr, 0.0)), np.maximum(fl, fr))
        else:
            sides = []
            for x in (left, right):
                u = np.concatenate([x[:1], x[:1] * x[1:-1], (x[-1:] / (gam - 1.0) + 0.5 * x[:1] * (x[1:-1] ** 2).sum(axis=0))])
                v = x[1 + k]
                fx = u * v
                fx[1 + k] += x[-1]
                fx[-1] += x[-1] * v
                sides.append((u, fx, v, np.sqrt(gam * x[-1] / x[0])))
            (ul, fl, vl, cl), (ur, fr, vr, cr) = sides
            sl, sr = np.minimum(vl - cl, vr - cr), np.maximum(vl + cl, vr + cr)
            with np.errstate(divide="ignore", invalid="ignore"):
                mid = (sr * fl - sl * fr + sl * sr * (ur - ul)) / (sr - sl)
            f = np.where(sl >= 0.0, fl, np.where(sr <= 0.0, fr, mid))
        out += np.moveaxis(-np.diff(f, axis=-1) / h, -1, ax)
    return out


def exact(case, seed):
    """The full-grid solves, by plain numpy.  Adaptive solves have none: a second implementation of the adaptive method
    in plain numpy would take minutes for each."""
    if case["kind"] != "solve" or case["adapt"] != "never" or case["time"] != "gts" or case["precision"] != "fp64" \
            or case["problem"] not in ("burgers1d", "burgers2d", "euler2d"):
        return None
    p, q, t_end = _make(case, random.Random(seed))
    nit, t = 1 << (p.max_level - p.min_level), 0.0
    while t < t_end:
        dt = p.cfl * 0.5 ** p.max_level / _speed(p, q)
        last = t + nit * dt >= t_end * (1.0 - 1e-14)
        if last:
            dt = (t_end - t) / nit
        for _ in range(nit):
            a = q + dt * _rhs(p, q)
            if p.rk_order == 2:
                q = 0.5 * q + 0.5 * a + 0.5 * dt * _rhs(p, a)
            else:
                b = 0.75 * q + 0.25 * a + 0.25 * dt * _rhs(p, a)
                q = q / 3.0 + 2.0 / 3.0 * b + 2.0 / 3.0 * dt * _rhs(p, b)
        t = t_end if last else t + nit * dt
    if case["read"] == "uniform":
        return q
    values = _room(p)[1]
    values[: q[0].size] = q.reshape(p.nvars(), -1).T
    return None, values
