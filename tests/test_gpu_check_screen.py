"""plan_check's FP32 screen never changes the FP64 minima: clearances against
plain FP64 over all pairs and walls, on plans whose closest pairs tie to
rounding (a rigid march), cross walls, or sit far from the origin, at agent
counts around a tile's edge."""
import math

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _seg(px, py, ax, ay, bx, by):
    dx, dy = bx - ax, by - ay
    dd = dx * dx + dy * dy
    t = np.clip(np.where(dd > 0, ((px - ax) * dx + (py - ay) * dy) / np.where(dd > 0, dd, 1), 0), 0, 1)
    return np.hypot(ax + t * dx - px, ay + t * dy - py)


def _clearances(z, r, walls):
    p = z.shape[0]
    i, j = np.triu_indices(p, 1)
    a, b = z[j, :-1] - z[i, :-1], z[j, 1:] - z[i, 1:]
    pair = (_seg(0.0, 0.0, a[..., 0], a[..., 1], b[..., 0], b[..., 1]) / (r[i] + r[j])[:, None]).min() if p > 1 else math.inf
    wall = math.inf
    for x0, y0, x1, y1 in walls:
        a, b = z[:, :-1], z[:, 1:]
        d = np.minimum(np.minimum(_seg(a[..., 0], a[..., 1], x0, y0, x1, y1), _seg(b[..., 0], b[..., 1], x0, y0, x1, y1)),
                       np.minimum(_seg(x0, y0, a[..., 0], a[..., 1], b[..., 0], b[..., 1]),
                                  _seg(x1, y1, a[..., 0], a[..., 1], b[..., 0], b[..., 1])))
        c = lambda u, v: u[..., 0] * v[..., 1] - u[..., 1] * v[..., 0]
        w0, w1 = np.array([x0, y0]), np.array([x1, y1])
        cross = (c(b - a, w0 - a) * c(b - a, w1 - a) < 0) & (c(w1 - w0, a - w0) * c(w1 - w0, b - w0) < 0)
        wall = min(wall, (np.where(cross, 0.0, d) / r[:, None]).min())
    return pair, wall


@pytest.mark.parametrize("p,eta,shift,march", [(1, 3, 0.0, False), (2, 1, 0.0, False), (32, 4, 0.0, True), (33, 4, 3000.0, True),
                                               (65, 3, 0.0, False), (200, 2, 100.0, True)])
def test_clearances_match_plain_fp64(p, eta, shift, march):
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(p, eta, seed=80 + p)
    rng = np.random.default_rng(p)
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    start, walls = f32(inst.start + shift), f32(inst.walls + shift)
    with pk.Planner(start, f32(inst.goal + shift), inst.radius, eta, walls=walls) as pl:
        r = f32(inst.radius)
        if march:  # every pair keeps its distance over every segment, to FP32 rounding
            z = start[:, None] + np.arange(eta + 1)[None, :, None] * 0.37
        else:      # crowded, crossing walls and each other
            z = start[:, None] + rng.normal(0, 0.5, size=(p, eta + 1, 2)) * np.arange(eta + 1)[None, :, None]
        z = f32(z)
        P = p * (p - 1) // 2
        pl.import_state(z, np.zeros((eta, P, 4, 2)), np.zeros((eta, p, 2, 2)), np.zeros((4, eta, p, 2, 2)), 0)
        got = [pl.check() for _ in range(2)]
    pair, wall = _clearances(z, r, walls)
    for g in got:  # the same FP64 arithmetic on the same FP32 values, in another order
        assert g["min_pair_clearance"] == pytest.approx(pair, rel=1e-13) if math.isfinite(pair) else math.isinf(g["min_pair_clearance"])
        assert g["min_wall_clearance"] == pytest.approx(wall, rel=1e-12, abs=1e-12 * (1 + shift))


@pytest.mark.parametrize("p,eta,far", [(300, 2, 0.0), (513, 1, 0.0), (70, 2, 1e12), (70, 2, 1e17)])
def test_bounding_circles_drop_no_closest_pair(p, eta, far):
    """Sparse plans, where the first bound drops nearly every block of pairs
    (the closest pair is planted in two groups, the bound comes from others),
    and an agent beyond the range of FP32 squares, where nothing may be dropped."""
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(p, eta, seed=180 + p)
    rng = np.random.default_rng(p)
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    with pk.Planner(f32(inst.start), f32(inst.goal), inst.radius, eta, walls=inst.walls) as pl:
        z = f32(inst.start[:, None] + rng.normal(0, 0.02, size=(p, eta + 1, 2)))
        z[p - 1, eta] = f32(z[1, eta] + 0.11 * inst.radius[1])
        if far:
            z[p // 2, :, 0] = np.float32(far)
        P = p * (p - 1) // 2
        pl.import_state(z, np.zeros((eta, P, 4, 2)), np.zeros((eta, p, 2, 2)), np.zeros((4, eta, p, 2, 2)), 0)
        got = [pl.check() for _ in range(2)]
    pair, _ = _clearances(z, f32(inst.radius), np.zeros((0, 4)))
    for g in got:  # the same FP64 arithmetic on the same FP32 values, in another order
        assert g["min_pair_clearance"] == pytest.approx(pair, rel=1e-13)
