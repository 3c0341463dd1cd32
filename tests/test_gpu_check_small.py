"""plan_check at the small end of FP32: motions shorter than its squares
resolve, and plans of sizes from 1e-6 to 1e-18."""
import numpy as np
import pytest

import workloads
from test_gpu_check_screen import _clearances

pytestmark = pytest.mark.gpu


def _check(inst, z, radius, walls):
    import paper_1311_4527_gb300 as pk
    p, eta = z.shape[0], z.shape[1] - 1
    with pk.Planner(inst.start, inst.goal, radius, eta, walls=walls) as pl:
        P = p * (p - 1) // 2
        pl.import_state(z, np.zeros((eta, P, 4, 2)), np.zeros((eta, p, 2, 2)), np.zeros((len(walls), eta, p, 2, 2)), 0)
        got = pl.check()
    return got["min_pair_clearance"], got["min_wall_clearance"]


@pytest.mark.parametrize("noise", [1e-18, 1e-21, 1e-23, 1e-30])
def test_noise_across_a_standing_agent_hides_no_pair(noise):
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    inst = workloads.small_square(4, 2, seed=9)
    z = np.zeros((4, 3, 2))
    z[1, :, 0], z[1, :, 1] = 1.0, [-noise, noise, -noise]   # passes agent 0 sideways, by nothing
    z[2, :, 0] = z[3, :, 0] = 10.0
    z[3, :, 1] = 0.5                                        # the closest pair
    z = f32(z)
    wall = f32([[-3.0, 0.0, -3.0, 1.0], [1.5, -noise, 1.5, noise]])
    pair, near = _check(inst, z, inst.radius, wall)
    want = _clearances(z, f32(inst.radius), wall)
    assert pair == pytest.approx(want[0], rel=1e-13) and near == pytest.approx(want[1], rel=1e-12)


@pytest.mark.parametrize("size", [2.0 ** -20, 2.0 ** -40, 2.0 ** -50, 2.0 ** -60])
def test_small_plans_are_checked_like_large_ones(size):
    f32 = lambda a: np.asarray(a, np.float32).astype(np.float64)
    inst = workloads.small_square(70, 2, seed=11)
    rng = np.random.default_rng(3)
    z = f32(inst.start[:, None] + rng.normal(0, 0.1, (70, 3, 2)))
    walls, r = f32(inst.walls), f32(inst.radius)
    one = _check(inst, z, r, walls)
    inst.start, inst.goal = f32(inst.start) * size, f32(inst.goal) * size
    got = _check(inst, z * size, r * size, walls * size)
    assert one[0] == pytest.approx(_clearances(z, r, walls)[0], rel=1e-13)
    assert got == pytest.approx(one, rel=1e-13)
