"""Iterates of circle swaps, with and without a speed limit, against stored
ones, to the bit: the minimizers' order of operations, fused or not, is part of
the results (csrc/twa_math.cuh), whichever kernel runs them."""
import json
import os

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "iterates.json")) as f:
    CASES = json.load(f)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "p%d" % c["p"])
def test_iterates_are_the_stored_ones(case):
    import paper_1311_4527_gb300 as pk
    inst = workloads.circle_swap(case["p"], case["eta"], 0.05, 0.02, case["seed"])
    kw = {"vmax": case["vmax"]} if case["vmax"] else {}
    with pk.Planner.from_instance(inst, **kw) as pl:
        pl.iterate(case["iterations"])
        z = pl.trajectory().cpu().numpy().reshape(-1)
    assert np.array_equal(z, np.asarray(case["z"], np.float32))
