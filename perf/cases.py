"""What is timed: the work a user of the planner has it do, through the public
entry points of ``paper_1311_4527_gb300``.

Every case is one pass: a plan re-solved for a fixed number of iterations, a
step of a control loop, an epoch of the local planner, a batch advanced, a
gradient, a final check.  Iteration counts are fixed budgets, so that a pass
is the same amount of work on every run, and short where the plan is crowded:
there a pair within rounding of touching changes which factors are weighted,
and long runs of two equally exact programs part.  ``exact`` is the same pass in 64-bit
torch, written from the method (App. B steps 1-7 of Bento et al., NIPS 2013).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1311_4527_gb300 as pk

# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------


def listed():
    return [
        # The smallest plan: four agents swap places on a circle.  A bounded
        # solve; the residual is read every 25 iterations.  Latency only.
        dict(name="swap4_solve", kind="solve", layout="circle", p=4, eta=4, r_lo=0.15, r_hi=0.15,
             jitter=0.01, rho0=1.0, iters=100),
        # An ordinary small plan: 100 robots of uneven size swap places.
        dict(name="swap100_solve", kind="solve", layout="circle", p=100, eta=8, r_lo=0.02, r_hi=0.05,
             jitter=0.02, rho0=2.0, iters=25),
        # Robots with a speed limit: a velocity factor per agent and segment.
        dict(name="swap48_speed_limit", kind="solve", layout="circle", p=48, eta=6, r_lo=0.02, r_hi=0.05,
             jitter=0.02, rho0=1.0, iters=50, vmax=0.4),
        # The benchmark's plan: 1024 agents in a walled square, 8.4 M collision
        # factors an iteration.
        dict(name="square1024", kind="iterate", layout="square", p=1024, eta=16, r_lo=0.2, r_hi=0.4,
             rho0=1.0, iters=4),
        # The largest plan, at an agent count that fills no tile: 134 M
        # collision factors an iteration.
        dict(name="square4095", kind="iterate", layout="square", p=4095, eta=16, r_lo=0.2, r_hi=0.4,
             rho0=1.0, iters=2),
        # Static obstacles: 64 interior walls beside the square's four sides.
        dict(name="obstacles300", kind="iterate", layout="square", p=300, eta=8, r_lo=0.2, r_hi=0.4,
             rho0=1.0, iters=8, obstacles=64),
        # The paper's baseline, standard ADMM, which updates the u of every
        # collision factor (the dense state).
        dict(name="admm512", kind="iterate", layout="square", p=512, eta=16, r_lo=0.2, r_hi=0.4,
             rho0=1.0, iters=16, mode="admm"),
        # Re-planning in a control loop: new endpoints from pinned host memory,
        # one iteration, the trajectory back to pinned host memory.
        dict(name="replan1024", kind="replan", layout="square", p=1024, eta=16, r_lo=0.2, r_hi=0.4,
             rho0=1.0, iters=1),
        # Many uneven plans at once, as for a sweep or a training set.
        dict(name="batch64", kind="batch", n=64, p_lo=8, p_hi=64, iters=4, tuned=True),
        # The gradient of a trajectory loss through 128 unrolled iterations.
        dict(name="gradient64", kind="gradient", layout="circle", p=64, eta=8, r_lo=0.02, r_hi=0.02,
             jitter=0.02, rho0=1.0, iters=128),
        # One epoch of the velocity-obstacle local planner for 32 robots about
        # to meet, with a fixed iteration budget.
        dict(name="epoch32", kind="epoch", p=32, iters=200),
        # The 64-bit feasibility and cost check of a finished plan.
        dict(name="check1024", kind="check", layout="march", p=1024, eta=16, r_lo=0.2, r_hi=0.4,
             rho0=1.0, iters=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "iterate", "iterate", "iterate", "admm", "replan", "batch", "gradient",
                       "epoch", "check"])
    if kind == "solve":
        c = dict(kind="solve", layout="circle", p=_log_int(rng, 2, 100), eta=rng.randint(2, 16), r_lo=0.02,
                 r_hi=0.05, jitter=0.02, rho0=rng.choice([0.5, 1.0, 2.0]), iters=25)
        if rng.random() < 0.3:
            c["vmax"] = 0.4
        return c
    if kind == "batch":
        return dict(kind="batch", n=_log_int(rng, 8, 64), p_lo=rng.randint(2, 16), p_hi=rng.randint(24, 64),
                    iters=rng.randint(2, 4), tuned=rng.random() < 0.5)
    if kind == "epoch":
        return dict(kind="epoch", p=_log_int(rng, 4, 128), iters=rng.choice([100, 200]))
    if kind == "gradient":
        return dict(kind="gradient", layout="circle", p=_log_int(rng, 4, 64), eta=rng.randint(2, 8), r_lo=0.02,
                    r_hi=0.02, jitter=0.02, rho0=1.0, iters=rng.randint(16, 128))
    square = dict(layout="square", eta=rng.randint(2, 16), r_lo=0.2, r_hi=0.4, rho0=1.0)
    if kind == "admm":
        mode = rng.choice(["admm", "dense"])
        return dict(square, kind="iterate", p=_log_int(rng, 16, 512), iters=rng.randint(4, 16 if mode == "admm" else 6),
                    mode=mode)
    if kind == "replan":
        return dict(square, kind="replan", p=_log_int(rng, 16, 2048), iters=rng.randint(1, 2))
    if kind == "check":
        return dict(square, kind="check", layout="march", p=_log_int(rng, 16, 1024), iters=0)
    c = dict(square, kind="iterate", p=_log_int(rng, 16, 4096))
    c["iters"] = 2 if c["p"] > 1024 else rng.randint(2, 6)
    if c["p"] <= 512 and rng.random() < 0.5:
        c["obstacles"] = rng.randint(1, 64)
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
# Circle swaps: agents evenly on a circle, goals at the antipodes, both a
# little off their places.  Squares: starts and goals placed at
# random without overlap, about 18 % of the area covered, the square's sides
# as walls, interior walls where asked for; in a march the goals are the
# starts moved by a quarter of the side, one way for all.


def _circle(p, radius, jitter, rng):
    ang = 2.0 * math.pi * np.arange(p) / p
    need = float(np.max(radius + np.roll(radius, -1))) if p > 1 else 0.0
    gap = max(1.25 * need, 1.02 * need + 3.0 * jitter)  # the jitter may not make neighbours touch
    rc = max(1.0, gap / (2.0 * math.sin(math.pi / p))) if p > 1 else 1.0
    at = rc * np.stack([np.cos(ang), np.sin(ang)], axis=1)
    off = rng.uniform(-jitter, jitter, size=(2, p, 2))
    return at + off[0], off[1] - at


def _place(rng, r, side, walls):
    """Disks of radius r one after another at random, none touching another
    (by 1 % of the radii) or an interior (axis-aligned) wall."""
    p = len(r)
    pos = np.full((p, 2), 1e9)
    lo, hi = np.minimum(walls[:, :2], walls[:, 2:]), np.maximum(walls[:, :2], walls[:, 2:])
    for i in range(p):
        for _ in range(100000):
            c = rng.uniform(1.01 * r[i], side - 1.01 * r[i], size=2)
            d = pos[:i] - c
            if i and np.any((d * d).sum(1) < (1.01 * (r[:i] + r[i])) ** 2):
                continue
            if len(walls) and np.any(((np.clip(c, lo, hi) - c) ** 2).sum(1) < (1.01 * r[i]) ** 2):
                continue
            pos[i] = c
            break
        else:
            raise RuntimeError("no room for every agent")
    return pos


def _interior_walls(rng, n, side):
    half = 0.5 * rng.uniform(side / 8, side / 4, size=n)
    c = rng.uniform(0.1 * side, 0.9 * side, size=(n, 2))
    flat = rng.uniform(size=n) < 0.5
    d = np.stack([np.where(flat, half, 0.0), np.where(flat, 0.0, half)], axis=1)
    return np.concatenate([c - d, c + d], axis=1)


def _instance(case, rng):
    p, eta = case["p"], case["eta"]
    r = rng.uniform(case["r_lo"], case["r_hi"], size=p)
    if case["layout"] == "circle":
        start, goal = _circle(p, r, case["jitter"], rng)
        walls = np.zeros((0, 4))
    else:
        side = math.sqrt(p * math.pi * np.mean(r * r) / 0.18) + 4 * case["r_hi"]
        inner = _interior_walls(rng, case.get("obstacles", 0), side)
        start = _place(rng, r, side, inner)
        if case["layout"] == "march":  # everyone moves the same way
            step = 0.25 * side
            goal, side = start + step, side + step
        else:
            goal = _place(rng, r, side, inner)
        walls = np.concatenate([[[0, 0, side, 0], [side, 0, side, side], [side, side, 0, side],
                                 [0, side, 0, 0]], inner]) if case.get("sides", True) else inner
    f32 = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)  # what the planner is given
    return SimpleNamespace(p=p, eta=eta, T=1.0, start=f32(start), goal=f32(goal), radius=f32(r),
                           cost_w=np.ones(p), walls=f32(walls), n_walls=len(walls), rho0=float(case["rho0"]),
                           alpha=0.1, tol=1e-6, max_iter=20000)


def _batch_members(case, rng):
    """Uneven members, circle swap or open square, as for a parameter sweep."""
    out = []
    sizes = np.random.default_rng([case["n"], case["p_lo"], case["p_hi"]])
    for _ in range(case["n"]):
        c = dict(p=int(sizes.integers(case["p_lo"], case["p_hi"] + 1)), eta=int(sizes.choice([4, 8, 16])),
                 r_lo=0.02, r_hi=0.05, rho0=1.0)
        c.update(dict(layout="circle", jitter=0.02) if sizes.uniform() < 0.5 else
                 dict(layout="square", sides=False))
        out.append(_instance(c, rng))
    return out


def _epoch_instance(case, rng):
    """Robots that have reached a tight ring on their way to the antipodes of
    a circle: neighbours are within a step of one another."""
    p = case["p"]
    r = np.full(p, 0.05)
    ring, far = _circle(p, r, 0.005, rng)
    size = 1.2 * 0.1 / (2.0 * math.sin(math.pi / p))  # 20 % more room than the disks take
    now = ring * (size / np.hypot(*far[0]))
    now = now.astype(np.float32)
    return SimpleNamespace(p=p, now=now, dest=far.astype(np.float32), radius=r,
                           c=(1.0 + 0.001 * np.arange(p)).astype(np.float32), step=0.1, advance=0.5,
                           rho0=30.0, alpha=0.5)


def _pinned(a):
    t = torch.empty(a.shape, dtype=torch.float32).pin_memory()
    t.copy_(torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)))
    return t.numpy(), t


def _flags(case):
    return {"admm": pk.PLAN_ADMM, "dense": pk.PLAN_DENSE_STATE}.get(case.get("mode"), 0)


def prepare(case, seed):
    rng = np.random.default_rng([seed, 1311])
    s = SimpleNamespace(case=case, K=case["iters"])
    kind = case["kind"]
    if kind == "batch":
        s.members = _batch_members(case, rng)
        s.batch = pk.PlannerBatch(s.members)
        if case["tuned"]:
            s.batch.set_shape(32, 4, 8)  # what the autotuner chooses for such a batch
        return s
    if kind == "epoch":
        i = _epoch_instance(case, rng)
        s.now = i.now
        s.plan = pk.Planner.velocity_obstacle(i.now, i.dest, i.radius, i.c, i.step, rho0=i.rho0, alpha=i.alpha,
                                              tol=1e-9, max_iter=s.K, check_every=50)
        return s
    inst = _instance(case, rng)
    kw = {"vmax": case["vmax"]} if "vmax" in case else {}
    # the budget ends a bounded solve, not the tolerance
    s.plan = pk.Planner.from_instance(inst, flags=_flags(case), check_every=25, tol=1e-9, max_iter=s.K, **kw)
    if kind == "replan":
        s.keep, s.at, s.turn = [], [], 0
        for start, goal in _replan_endpoints(inst):
            a, b = _pinned(start), _pinned(goal)
            s.keep += [a[1], b[1]]
            s.at.append((a[0], b[0]))
        s.out, t = _pinned(np.zeros((inst.p, inst.eta + 1, 2)))
        s.keep.append(t)
    elif kind == "gradient":
        dev = s.plan.device
        t = lambda a: torch.tensor(a, dtype=torch.float32, device=dev, requires_grad=True)
        s.args = [t(inst.start), t(inst.goal), t(inst.radius), t(inst.cost_w)]
        s.gz = torch.tensor(_loss_gradient(inst, rng), dtype=torch.float32, device=dev)
    elif kind == "check":
        P = inst.p * (inst.p - 1) // 2
        s.plan.import_state(_march(inst, rng), np.zeros((inst.eta, P, 4, 2), np.float32),
                            np.zeros((inst.eta, inst.p, 2, 2)), np.zeros((inst.n_walls, inst.eta, inst.p, 2, 2)), 1)
    return s


def _replan_endpoints(inst):
    """Two sets of measured positions: everyone a little off."""
    d = 0.004 * float(np.min(inst.radius))
    return [((inst.start + k * d).astype(np.float32), (inst.goal - k * d).astype(np.float32)) for k in (0.5, -0.5)]


def _march(inst, rng):
    """A finished plan's break-points: a march from the starts to the goals,
    a little uneven (the starts leave 1 % of the radii between the agents)."""
    t = np.arange(inst.eta + 1)[None, :, None] / inst.eta
    z = inst.start[:, None] + t * (inst.goal - inst.start)[:, None]
    z[:, 1:-1] += rng.uniform(-0.002, 0.002, size=z[:, 1:-1].shape) * inst.radius[:, None, None]
    z[:, -1] = inst.goal
    return z.astype(np.float32)


def _loss_gradient(inst, rng):
    """dL/dz of a trajectory loss (a tracking error: every break-point but the fixed ends)."""
    g = rng.normal(size=(inst.p, inst.eta + 1, 2))
    g[:, 0] = 0.0
    g[:, -1] = 0.0
    return g.astype(np.float32)


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------


def run(s):
    kind = s.case["kind"]
    if kind == "solve":
        s.plan.reset()
        done, iterations, _ = s.plan.solve()
        return {"z": s.plan.trajectory(), "done": done, "iterations": iterations}
    if kind == "iterate":
        s.plan.reset()
        s.plan.iterate(s.K)
        return {"z": s.plan.trajectory()}
    if kind == "replan":
        start, goal = s.at[s.turn]
        s.turn ^= 1
        s.plan.set_endpoints(start, goal, wait=False)
        s.plan.iterate(s.K)
        return {"z": s.plan.trajectory_host(s.out)}
    if kind == "batch":
        s.batch.iterate(s.K)
        return {"z": torch.cat([s.batch.trajectory(b).reshape(-1) for b in range(s.batch.n)])}
    if kind == "epoch":
        s.plan.set_endpoints(s.now, s.now)
        done, iterations, _, far = s.plan.vo_epoch(0.5)
        x0, ref = s.plan.endpoints()
        return {"z": s.plan.trajectory(), "x0": x0, "ref": ref, "far": far, "done": done,
                "iterations": iterations}
    if kind == "gradient":
        for a in s.args:
            a.grad = None
        z = pk.unrolled_trajectory(s.plan, *s.args, s.K)
        z.backward(s.gz)
        return {"z": z.detach(), "start": s.args[0].grad, "goal": s.args[1].grad, "radius": s.args[2].grad,
                "cost": s.args[3].grad}
    c = s.plan.check()
    return {k: np.float64(c[k]) for k in ("total_cost", "min_pair_clearance", "min_wall_clearance",
                                          "max_endpoint_error")}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------


def work(case):
    """Bytes: inputs and state read once, results and state written once.
    Operations: per iteration, a relative-motion test of every pair and
    segment (about 12), about 40 a kinetic factor, 20 an agent-wall test; with
    the dense state every u record moves too (32 bytes in, 32 out, per factor
    and iteration, where the records of all factors do not fit on the chip)."""
    kind, K = case["kind"], case["iters"]
    if kind == "batch":
        pm = (case["p_lo"] + case["p_hi"]) / 2
        pp = (case["p_lo"] ** 2 + case["p_lo"] * case["p_hi"] + case["p_hi"] ** 2) / 3
        eta = 28 / 3
        return {"bytes": case["n"] * pm * (8 * eta * 6 + 40), "flops": case["n"] * K * eta * (6 * pp + 40 * pm)}
    p, eta = case["p"], case.get("eta", 2)
    nw = case.get("obstacles", 0) + (4 if case.get("layout") in ("square", "march") else 0)
    pairs, segs = p * (p - 1) / 2, (1 if kind == "epoch" else eta)
    per = segs * pairs * 12 + eta * p * 40 + segs * p * nw * 20
    state = p * (eta + 1) * 8 + eta * p * 32
    if kind == "check":
        return {"bytes": p * (eta + 1) * 8, "flops": per}
    if case.get("mode"):
        dense = eta * pairs * 32
        return {"bytes": 2 * state + K * 2 * dense if dense > 100e6 else 2 * (state + dense), "flops": K * per}
    if kind == "gradient":  # the iteration, and an adjoint of about twice its factors' work
        return {"bytes": 4 * state, "flops": K * (per + 2 * eta * p * 40)}
    return {"bytes": 2 * state, "flops": K * per}


# --------------------------------------------------------------------------
# the same pass in 64 bits
# --------------------------------------------------------------------------


def _dot(a, b):
    return (a * b).sum(-1)


def _turn(n):
    return torch.stack([-n[..., 1], n[..., 0]], -1)


def _unit(t):
    return torch.stack([torch.cos(t), torch.sin(t)], -1)


def _seg_dist(p0, p1):
    """Distance of the origin from the segments [p0, p1]."""
    d = p1 - p0
    dd = _dot(d, d)
    t = torch.where(dd > 0, -_dot(p0, d) / torch.where(dd > 0, dd, torch.ones_like(dd)), torch.zeros_like(dd))
    return (p0 + t.clamp(0, 1)[..., None] * d).norm(dim=-1)


def _wall_dist(a0, a1, c0, c1):
    """Distance between the segments [a0, a1] and [c0, c1]."""
    m = torch.minimum(torch.minimum(_seg_dist(c0 - a0, c1 - a0), _seg_dist(c0 - a1, c1 - a1)),
                      torch.minimum(_seg_dist(a0 - c0, a1 - c0), _seg_dist(a0 - c1, a1 - c1)))
    x = lambda u, v: u[..., 0] * v[..., 1] - u[..., 1] * v[..., 0]
    cross = (x(a1 - a0, c0 - a0) * x(a1 - a0, c1 - a0) < 0) & (x(c1 - c0, a0 - c0) * x(c1 - c0, a1 - c0) < 0)
    return torch.where(cross, torch.zeros_like(m), m)


def _hinges(t, a, b, c0, c1, r):
    """At direction t: each end's shortfall from the region's support, and
    its position along t and across it, seen from the supporting end."""
    n = _unit(t)
    k = _turn(n)
    second = _dot(c1, n) > _dot(c0, n)
    c = torch.where(second[..., None], c1, c0)
    an, bn = _dot(a - c, n), _dot(b - c, n)
    return (r - an).clamp_min(0), (r - bn).clamp_min(0), an, bn, _dot(a - c, k), _dot(b - c, k)


def _energy(t, a, b, c0, c1, r):
    ga, gb = _hinges(t, a, b, c0, c1, r)[:2]
    return 0.5 * (ga * ga + gb * gb)


def _slope(t, a, b, c0, c1, r):
    """dE/dt and d2E/dt2 away from a kink of the support."""
    ga, gb, an, bn, at, bt = _hinges(t, a, b, c0, c1, r)
    e1 = -(ga * at + gb * bt)
    e2 = (ga > 0) * (at * at + ga * an) + (gb > 0) * (bt * bt + gb * bn)
    return e1, e2


@torch.no_grad()
def _best_free(a, b, c0, c1, r, grid=360, keep=6):
    """Angle of the separating direction of least energy, both ends free with
    equal weights: a scan, then golden section in the best valleys, then
    Newton where the energy is smooth."""
    out = torch.zeros_like(r)
    kink = torch.zeros_like(r, dtype=torch.bool)
    for at in range(0, len(r), 32768):
        q = slice(at, at + 32768)
        A, B, C0, C1, R = a[q], b[q], c0[q], c1[q], r[q]
        step = 2 * math.pi / grid
        t = torch.arange(grid, dtype=torch.float64, device=r.device) * step
        w = lambda v: v[:, None]
        e = _energy(t[None], w(A), w(B), w(C0), w(C1), w(R))
        valley = (e <= e.roll(1, 1)) & (e <= e.roll(-1, 1))
        k = torch.where(valley, e, torch.full_like(e, math.inf)).topk(keep, 1, largest=False).indices
        lo, hi = t[k] - step, t[k] + step
        g = (math.sqrt(5) - 1) / 2
        for _ in range(44):
            m1, m2 = hi - g * (hi - lo), lo + g * (hi - lo)
            left = _energy(m1, w(A), w(B), w(C0), w(C1), w(R)) <= _energy(m2, w(A), w(B), w(C0), w(C1), w(R))
            hi, lo = torch.where(left, m2, hi), torch.where(left, lo, m1)
        c = 0.5 * (lo + hi)
        for _ in range(4):
            e1, e2 = _slope(c, w(A), w(B), w(C0), w(C1), w(R))
            d = torch.where(e2 > 0, -e1 / torch.where(e2 > 0, e2, torch.ones_like(e2)), torch.zeros_like(e2))
            better = _energy(c + d, w(A), w(B), w(C0), w(C1), w(R)) <= _energy(c, w(A), w(B), w(C0), w(C1), w(R))
            c = torch.where((d.abs() < 1e-5) & better, c + d, c)
        along = C1 - C0
        kt = torch.atan2(along[:, 0], -along[:, 1])  # the wall's normals, where its two ends support alike
        c = torch.cat([c, kt[:, None], kt[:, None] + math.pi], 1)
        best = _energy(c, w(A), w(B), w(C0), w(C1), w(R)).argmin(1)
        out[q] = c.gather(1, best[:, None])[:, 0]
        kink[q] = best >= keep
    return out, kink


def _free_ends(a, b, c0, c1, r):
    """Ends of the cheapest segment that clears the region, both ends free."""
    t, kink = _best_free(a.detach(), b.detach(), c0.detach(), c1.detach(), r.detach())
    if torch.is_grad_enabled():
        # the minimum moves with its inputs: one Newton step, whose value is zero
        e1, e2 = _slope(t, a, b, c0, c1, r)
        ok = (e2.detach() > 1e-9) & ~kink
        t = t - torch.where(ok, e1 / torch.where(ok, e2.detach(), torch.ones_like(e2)), torch.zeros_like(e1))
    n = _unit(t)
    h = torch.maximum(_dot(c0, n), _dot(c1, n)) + r
    lift = lambda v: v + (h - _dot(v, n)).clamp_min(0)[..., None] * n
    return lift(a), lift(b)


def _fixed_end(q, w, c0, c1, r):
    """The free end nearest to w, the other end held at q."""
    cand = []
    for c in (c0, c1):
        v = q - c
        off = torch.acos((r / v.norm(dim=-1).clamp_min(1e-300)).clamp(-1, 1))
        base = torch.atan2(v[:, 1], v[:, 0])
        u = w - c
        cand += [base + off, base - off, torch.atan2(u[:, 1], u[:, 0])]
    along = c1 - c0
    k = torch.atan2(along[:, 0], -along[:, 1])
    t = torch.stack(cand + [k, k + math.pi], 1)
    with torch.no_grad():
        n = _unit(t)
        e = lambda v: v[:, None]
        h = torch.maximum(_dot(e(c0), n), _dot(e(c1), n)) + e(r)
        gap = (h - _dot(e(w), n)).clamp_min(0)
        clear = _dot(e(q), n) - h >= -1e-12 * (1 + q.abs().amax(1))[:, None]
        best = torch.where(clear, gap, torch.full_like(gap, math.inf)).argmin(1)
    n = _unit(t.gather(1, best[:, None])[:, 0])
    h = torch.maximum(_dot(c0, n), _dot(c1, n)) + r
    return w + (h - _dot(w, n)).clamp_min(0)[..., None] * n


def _clear(a, b, c0, c1, r, lo, hi):
    """Ends of the cheapest segment that clears the region; an end is held
    where lo / hi says so."""
    va, vb = a, b
    for held, f in ((~lo & ~hi, lambda m: _free_ends(a[m], b[m], c0[m], c1[m], r[m])),
                    (lo & ~hi, lambda m: (a[m], _fixed_end(a[m], b[m], c0[m], c1[m], r[m]))),
                    (hi & ~lo, lambda m: (_fixed_end(b[m], a[m], c0[m], c1[m], r[m]), b[m]))):
        m = held.nonzero()[:, 0]
        if len(m):
            x, y = f(m)
            va, vb = va.index_copy(0, m, x), vb.index_copy(0, m, y)
    return va, vb


class _Plan64:
    """The iteration in 64-bit torch, every factor's u kept."""

    def __init__(self, start, goal, radius, eta, cost, walls, rho, alpha, device, admm=False, vmax=None, vo=False):
        t = lambda v: v if torch.is_tensor(v) else torch.tensor(np.asarray(v), dtype=torch.float64, device=device)
        self.start, self.goal, self.radius, self.walls = t(start), t(goal), t(radius), t(walls)
        self.p, self.eta, self.rho, self.alpha = len(self.radius), eta, rho, alpha
        self.admm, self.vmax, self.vo = admm, vmax, vo
        self.c = t(cost)[:, None].expand(self.p, eta) / (1 if vo else self.p * eta)
        self.i, self.j = torch.triu_indices(self.p, self.p, 1, device=device)
        self.segs = [0] if vo else list(range(eta))
        f = dict(dtype=torch.float64, device=device)
        z = self.start[:, None].expand(self.p, eta + 1, 2)
        self.z = torch.cat([z[:, :eta], self.goal[:, None]], 1)
        self.u = {s: torch.zeros(len(self.i), 4, 2, **f) for s in self.segs}
        self.uk = torch.zeros(self.p, eta, 2, 2, **f)
        self.uw = torch.zeros(len(self.walls), self.p, eta, 2, 2, **f)
        self.uv = torch.zeros(self.p, eta, 2, 2, **f)

    def fix_ends(self, start, goal):
        self.start, self.goal = start, goal
        self.z = torch.cat([start[:, None], self.z[:, 1:-1], goal[:, None]], 1)

    def _kinetic(self, n):
        """Closed form per end weights: the fixed ends stay."""
        s = torch.arange(self.eta, device=n.device)
        lo, hi = (s == 0)[None, :, None], (s == self.eta - 1)[None, :, None]
        c, rho, a, b = self.c[..., None], self.rho, n[:, :, 0], n[:, :, 1]
        free = 4 * c + rho
        one = 2 * c + rho
        xa = torch.where(lo, a, torch.where(hi, (rho * a + 2 * c * b) / one, (rho * a + 2 * c * (a + b)) / free))
        xb = torch.where(hi, b, torch.where(lo, (rho * b + 2 * c * a) / one, (rho * b + 2 * c * (a + b)) / free))
        return torch.stack([xa, xb], 2)

    def iterate(self):
        p, eta, dev = self.p, self.eta, self.z.device
        E1 = eta + 1
        num = torch.zeros(p * E1, 2, dtype=torch.float64, device=dev)
        den = torch.zeros(p * E1, dtype=torch.float64, device=dev)
        edges = []  # (node, x, u before, where the new u goes)

        def send(node, x, u, put):
            nonlocal num, den
            num = num.index_add(0, node.reshape(-1), (x + u).reshape(-1, 2))
            den = den.index_add(0, node.reshape(-1), torch.ones(node.numel(), dtype=torch.float64, device=dev))
            edges.append((node, x, u, put))

        # kinetic factors (the local planner's run on the second segment only)
        ends = torch.stack([self.z[:, :-1], self.z[:, 1:]], 2)
        node = (torch.arange(p, device=dev)[:, None, None] * E1 + torch.arange(eta, device=dev)[None, :, None]
                + torch.arange(2, device=dev))
        x = self._kinetic(ends - self.uk)
        k0 = 1 if self.vo else 0
        send(node[:, k0:], x[:, k0:], self.uk[:, k0:],
             lambda v: setattr(self, "uk", torch.cat([self.uk[:, :k0], v], 1)))
        # collision factors: every segment's colliding pairs through one minimizer call
        flat, i, j, R = self.z.reshape(-1, 2), self.i, self.j, self.radius[self.i] + self.radius[self.j]
        found = []
        for s in self.segs:
            nodes = torch.stack([i * E1 + s, i * E1 + s + 1, j * E1 + s, j * E1 + s + 1], 1)
            n = flat[nodes] - self.u[s]
            hit = (_seg_dist(n[:, 2] - n[:, 0], n[:, 3] - n[:, 1]) < R).nonzero()[:, 0]
            found.append((s, hit, n[hit], nodes, n if self.admm else None))
        m = torch.cat([f[2] for f in found])
        at = torch.cat([torch.full_like(f[1], f[0]) for f in found])
        zero = torch.zeros(len(m), 2, dtype=torch.float64, device=dev)
        vl, vh = _clear(m[:, 2] - m[:, 0], m[:, 3] - m[:, 1], zero, zero, R[torch.cat([f[1] for f in found])],
                        at == 0, at == eta - 1)
        sl, sh = m[:, 0] + m[:, 2], m[:, 1] + m[:, 3]
        xs = torch.stack([0.5 * (sl - vl), 0.5 * (sh - vh), 0.5 * (sl + vl), 0.5 * (sh + vh)], 1)
        for (s, hit, _, nodes, n), x in zip(found, xs.split([len(f[1]) for f in found])):
            u = self.u[s]
            if self.admm:  # every factor is weighted; a feasible one returns its n
                send(nodes, n.index_copy(0, hit, x), u, lambda v, s=s: self.u.__setitem__(s, v))
            else:
                send(nodes[hit], x, u[hit],
                     lambda v, s=s, h=hit, u=u: self.u.__setitem__(s, torch.zeros_like(u).index_copy(0, h, v)))
        del found
        # walls, every wall's active factors through one minimizer call
        con = torch.tensor(self.segs, device=dev)
        if len(self.walls):
            n = ends - self.uw
            c0, c1 = (self.walls[:, None, None, k:k + 2] for k in (0, 2))
            d = _wall_dist(n[:, :, con, 0], n[:, :, con, 1], c0, c1)
            hit = d < self.radius[:, None]
            w, a, k = (torch.ones_like(hit) if self.admm else hit).nonzero(as_tuple=True)
            s = con[k]
            q, m = n[w, a, s], hit[w, a, k].nonzero()[:, 0]
            x0, x1 = _clear(q[m, 0], q[m, 1], self.walls[w[m], :2], self.walls[w[m], 2:], self.radius[a[m]],
                            s[m] == 0, s[m] == eta - 1)
            x = torch.stack([q[:, 0].index_copy(0, m, x0), q[:, 1].index_copy(0, m, x1)], 1)
            at = (w * p + a) * eta + s
            send(node[a, s], x, self.uw[w, a, s],
                 lambda v, at=at: setattr(self, "uw", torch.zeros_like(self.uw).reshape(-1, 2, 2)
                                          .index_copy(0, at, v).reshape(self.uw.shape)))
        # the speed limit
        if self.vmax is not None:
            n = (ends - self.uv)[:, con]
            d = n[:, :, 0] - n[:, :, 1]
            L = d.norm(dim=-1)
            a, k = (L > self.vmax).nonzero(as_tuple=True)
            s = con[k]
            q, g = n[a, k], (self.vmax / L[a, k])[:, None] * d[a, k]
            lo, hi = (s == 0)[:, None], (s == eta - 1)[:, None]
            mid = 0.5 * (q[:, 0] + q[:, 1])
            xl = torch.where(lo, q[:, 0], torch.where(hi, q[:, 1] + g, mid + 0.5 * g))
            xh = torch.where(hi, q[:, 1], torch.where(lo, q[:, 0] - g, mid - 0.5 * g))
            flat = a * eta + s
            send(node[a, s], torch.stack([xl, xh], 1), self.uv[a, s],
                 lambda v, f=flat: setattr(self, "uv", torch.zeros_like(self.uv).reshape(-1, 2, 2)
                                           .index_copy(0, f, v).reshape(p, eta, 2, 2)))
        # the mean of what arrives; the fixed ends stay
        zn = torch.where(den[:, None] > 0, num / den.clamp_min(1)[:, None], self.z.reshape(-1, 2)).reshape(p, E1, 2)
        zn = torch.cat([self.start[:, None], zn[:, 1:-1], self.goal[:, None]], 1)
        flat = zn.reshape(-1, 2)
        at = torch.arange(E1, device=dev).repeat(p)
        free = ((at > 0) & (at < eta))
        self.uv = torch.zeros_like(self.uv)
        for nd, x, u, put in edges:
            step = torch.where(free[nd][..., None], x - flat[nd], torch.zeros_like(x))
            put(torch.where(free[nd][..., None], u + self.alpha * step, torch.zeros_like(u)))
        self.z = zn


def _check(P, z):
    """Cost, smallest pair and wall clearance and endpoint error of break-points z."""
    pair, R = math.inf, P.radius[P.i] + P.radius[P.j]
    for s in range(P.eta if len(P.i) else 0):
        pair = min(pair, float((_seg_dist(z[P.j, s] - z[P.i, s], z[P.j, s + 1] - z[P.i, s + 1]) / R).min()))
    c0, c1 = (P.walls[:, None, None, k:k + 2] for k in (0, 2))
    wall = float((_wall_dist(z[:, :-1], z[:, 1:], c0, c1) / P.radius[:, None]).min())
    return {"total_cost": np.float64((P.c * ((z[:, 1:] - z[:, :-1]) ** 2).sum(-1)).sum().item()),
            "min_pair_clearance": np.float64(pair), "min_wall_clearance": np.float64(wall),
            "max_endpoint_error": np.float64(max((z[:, 0] - P.start).abs().max().item(),
                                                 (z[:, -1] - P.goal).abs().max().item()))}


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    rng = np.random.default_rng([seed, 1311])
    kind, K = case["kind"], case["iters"]
    if kind == "batch":
        if case["n"] * K > 500:
            return None  # too long
        zs = []
        with torch.no_grad():
            for i in _batch_members(case, rng):
                P = _Plan64(i.start, i.goal, i.radius, i.eta, i.cost_w, i.walls, i.rho0, i.alpha, dev)
                for _ in range(K):
                    P.iterate()
                zs.append(P.z.reshape(-1))
        return {"z": torch.cat(zs)}
    if kind == "epoch":
        i = _epoch_instance(case, rng)
        now, dest = (torch.tensor(v, dtype=torch.float64, device=dev) for v in (i.now, i.dest))
        d = dest - now
        L = d.norm(dim=-1, keepdim=True)
        ref = now + torch.where(L > i.step, i.step / L, torch.ones_like(L)) * d
        P = _Plan64(now, ref, i.radius.astype(np.float32).astype(np.float64), 2, i.c.astype(np.float64),
                    np.zeros((0, 4)), i.rho0, i.alpha, dev, vo=True)
        for _ in range(K):
            P.iterate()
        new = now + i.advance * (P.z[:, 1] - now)
        far = float((dest - new).norm(dim=-1).max())
        return {"z": P.z, "x0": new, "ref": ref, "far": far, "done": None, "iterations": None}
    inst = _instance(case, rng)
    make = lambda *a: _Plan64(*a, inst.walls, inst.rho0, inst.alpha, dev, admm=case.get("mode") == "admm",
                              vmax=float(np.float32(case["vmax"])) if "vmax" in case else None)
    if kind == "check":
        P = make(inst.start, inst.goal, inst.radius, inst.eta, inst.cost_w)
        return _check(P, torch.tensor(_march(inst, rng), dtype=torch.float64, device=dev))
    if kind == "gradient":
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev, requires_grad=True)
        args = [t(inst.start), t(inst.goal), t(inst.radius), t(inst.cost_w)]
        P = make(args[0], args[1], args[2], inst.eta, args[3])
        for _ in range(K):
            P.iterate()
        P.z.backward(torch.tensor(_loss_gradient(inst, rng), dtype=torch.float64, device=dev))
        return {"z": P.z.detach(), "start": args[0].grad, "goal": args[1].grad, "radius": args[2].grad,
                "cost": args[3].grad}
    with torch.no_grad():
        P = make(inst.start, inst.goal, inst.radius, inst.eta, inst.cost_w)
        if kind == "replan":
            start, goal = _replan_endpoints(inst)[0]
            P.fix_ends(*(torch.tensor(v, dtype=torch.float64, device=dev) for v in (start, goal)))
        for _ in range(K):
            P.iterate()
    return {"z": P.z, "done": None, "iterations": None} if kind == "solve" else {"z": P.z}
