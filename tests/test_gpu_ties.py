"""Gradients of circle swaps on whose way a candidate direction of the collision
minimizer ties with another one to rounding.  The winner decides the branch
that the adjoint differentiates, so any change of the minimizers' rounding
moves these gradients by 5e-5 and more (2-norm of a group, relative); the
stored values are those of the arithmetic that csrc/twa_math.cuh spells out."""
import json
import os

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "gradient_ties.json")) as f:
    CASES = json.load(f)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "p%d" % c["p"])
def test_gradients_at_ties_are_the_stored_ones(case):
    import torch
    import paper_1311_4527_gb300 as pk
    p, eta = case["p"], case["eta"]
    inst = workloads.circle_swap(p, eta, 0.02, 0.01, case["seed"])
    gz = np.random.default_rng(case["seed"]).normal(size=(p, eta + 1, 2)).astype(np.float32)
    gz[:, 0] = gz[:, -1] = 0
    with pk.Planner.from_instance(inst) as pl:
        args = [torch.tensor(v, dtype=torch.float32, device=pl.device, requires_grad=True)
                for v in (inst.start, inst.goal, inst.radius, inst.cost_w)]
        z = pk.unrolled_trajectory(pl, *args, case["iterations"])
        z.backward(torch.tensor(gz, device=pl.device))
        got = {"z": z.detach(), **{n: a.grad for n, a in zip(("start", "goal", "radius", "cost"), args)}}
    for name, v in got.items():
        # FP64 atomics may add up in another order: the last bits of FP32 adjoints, over 60 iterations
        want = np.asarray(case[name], np.float64)
        off = np.linalg.norm(v.cpu().numpy().astype(np.float64).reshape(-1) - want) / np.linalg.norm(want)
        assert off <= 5e-6, (name, off)
