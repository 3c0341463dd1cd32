"""Plans large enough for sorted tiles, on the ways that other tests take with
small plans only: an imported state, runs long enough for the graph of 64
iterations and the sort behind it, speed limits, the feasibility problem, and
the backward pass.  The dense state visits every pair and does not sort."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _z(pl):
    return pl.trajectory().cpu().numpy()


def test_an_imported_state_goes_on_like_its_own():
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(2880, 11, seed=51)
    with pk.Planner.from_instance(inst) as a, pk.Planner.from_instance(inst) as b:
        a.iterate(20)
        st = a.export_state()
        b.import_state(*(st[k].cpu().numpy() for k in ("z", "u_coll", "u_kin", "u_wall")), st["k"])
        del st
        for n in (1, 3, 20):
            a.iterate(n)
            b.iterate(n)
            assert np.array_equal(_z(a), _z(b)), n
            assert a.info()["active_coll"] == b.info()["active_coll"] > 0


@pytest.mark.parametrize("kw,runs", [({}, (1, 64 + 16 + 1, 9)), ({"vmax": 0.5}, (1, 20)), ({"energy": False}, (1, 20))])
def test_runs_equal_the_dense_state(kw, runs):
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(2047, 21, seed=52)
    out = []
    for flags in (0, pk.PLAN_DENSE_STATE):
        with pk.Planner.from_instance(inst, flags=flags, **kw) as pl:
            zs = []
            for n in runs:
                pl.iterate(n)
                zs.append((_z(pl), pl.info()["active_coll"]))
            out.append(zs)
    for (zg, ag), (zd, ad) in zip(*out):
        assert np.array_equal(zg, zd) and ag == ad > 0


def test_gradients_equal_the_dense_state():
    import torch
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(2047, 21, seed=53)
    gz = torch.randn(2047, 22, 2, generator=torch.Generator().manual_seed(1))
    out = []
    for flags in (0, pk.PLAN_DENSE_STATE):
        with pk.Planner.from_instance(inst, flags=flags) as pl:
            pl.unroll(5, 2)
            out.append([pl.trajectory()] + list(pl.backward(gz)) + [pl.trajectory()])
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][0], out[0][-1]) and torch.equal(out[1][0], out[1][-1])
    for a, b in zip(out[0][1:-1], out[1][1:-1]):
        # the same FP32 steps with FP64 sums in another order
        assert float((a - b).abs().max()) <= 1e-5 * float(b.abs().max())
