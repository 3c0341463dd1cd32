"""A wall that an agent's way crosses is active whatever the unit of length:
the test that leaves out walls out of reach may not overflow."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [2.0 ** -30, 1.0, 2.0 ** 28, 2.0 ** 31, 2.0 ** 34])
def test_a_crossed_wall_is_active(unit):
    import paper_1311_4527_gb300 as pk
    start, goal = np.array([[-1.8, 0.0]]) * unit, np.array([[0.2, 0.1]]) * unit
    walls = np.array([[0.0, -5.0, 0.0, 5.0], [9.0, -5.0, 9.0, 5.0]]) * unit
    with pk.Planner(start, goal, np.array([0.1]) * unit, 2, walls=walls) as pl:
        pl.iterate(1)
        act = pl.export_state()["act_wall"].cpu().numpy()
    assert act[0, 1, 0] == 1 and act[1].sum() == 0
