"""plan_check's wall clearance where FP32 cross products say that an agent far
away crosses a wall: agents that move along the line of an oblique wall beyond
its ends, beside one that violates it."""
import numpy as np
import pytest

import workloads
from test_gpu_check_screen import _clearances

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(12))
def test_agents_on_a_walls_line_hide_no_violation(seed):
    import paper_1311_4527_gb300 as pk
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    rng = np.random.default_rng(seed)
    p, eta = 120, 2
    inst = workloads.small_square(p, eta, seed=400 + seed)
    at, turn, half = rng.uniform(-5, 5, 2), rng.uniform(0, 2 * np.pi), rng.uniform(0.5, 2)
    along = np.array([np.cos(turn), np.sin(turn)])
    wall = f32(np.concatenate([at - half * along, at + half * along]))[None]
    # beyond the ends, on the line, in steps along it
    u = (half + rng.uniform(0.5, 3, (p, 1)) + np.cumsum(rng.uniform(0.1, 1, (p, eta + 1)), 1)) * rng.choice([-1, 1], (p, 1))
    z = at + u[..., None] * along
    # one agent beside the wall, at half its radius
    off = 0.5 * f32(inst.radius)[7] * np.array([-along[1], along[0]])
    z[7] = at + off + np.linspace(-0.4, 0.4, eta + 1)[:, None] * half * along
    z = f32(z)
    with pk.Planner(f32(inst.start) + 50, f32(inst.goal) + 50, inst.radius, eta, walls=wall) as pl:
        P = p * (p - 1) // 2
        pl.import_state(z, np.zeros((eta, P, 4, 2)), np.zeros((eta, p, 2, 2)), np.zeros((1, eta, p, 2, 2)), 0)
        got = pl.check()["min_wall_clearance"]
    want = _clearances(z, f32(inst.radius), wall)[1]
    assert want == pytest.approx(0.5, abs=1e-5)
    assert got == pytest.approx(want, rel=1e-12)
