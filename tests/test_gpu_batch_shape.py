"""The autotuner of a gated batch leaves the dense state's launch shapes as
they were set: no launch depends on them, so their timings differ by noise."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,ctas", [(4, 3), (16, 8), (32, 2)])
def test_shapes_without_effect_stay(rows, ctas):
    import paper_1311_4527_gb300 as pk
    with pk.PlannerBatch([workloads.circle4(), workloads.small_square(20, 4, seed=1)]) as batch:
        batch.set_shape(rows, ctas, 2)
        got = batch.autotune(2)
    assert got["rows_per_warp"] == rows and got["prox_ctas_per_sm"] == ctas
    assert got["iterations_per_graph"] in (2, 8)
