"""The gated state's factor pass (worklist, tile and segment warps) against
the dense state, which visits every pair and shares only the per-factor
arithmetic: the same iterates bit for bit, whatever made the worklist (a fresh
start, appends, rebuilds, an imported state), at agent counts on both sides of
a tile's edge and segment counts on both sides of a node warp's."""
import numpy as np
import pytest

import workloads
from oracle import twa

import _parity as par

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,eta,iters", [(2, 3, 40), (31, 2, 60), (32, 5, 60), (33, 4, 120), (65, 9, 120), (130, 3, 80)])
def test_gated_and_dense_iterates_are_bitwise_equal(p, eta, iters):
    import paper_1311_4527_gb300 as pk
    inst = workloads.circle_swap(p, eta, None, 0.005, 50 + p, radius_range=(0.02, 0.05))
    out = []
    for flags in (0, pk.PLAN_DENSE_STATE):
        with pk.Planner.from_instance(inst, flags=flags) as pl:
            zs = []
            for n in (1, 1, iters // 2, iters - iters // 2):
                r = pl.iterate(n, residual=True)
                zs.append((pl.trajectory().cpu().numpy(), r, pl.info()["active_coll"]))
        out.append(zs)
    assert out[0][-1][2] > 0 or p == 2
    for g, d in zip(*out):
        assert np.array_equal(g[0], d[0]) and g[1] == d[1] and g[2] == d[2]


def test_any_worklist_gives_the_same_iterates():
    """Iterations from a state whose worklist was appended to for a while and
    from the same state imported (worklist rebuilt from the activity bits)."""
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(70, 6, seed=23)
    with pk.Planner.from_instance(inst) as a, pk.Planner.from_instance(inst) as b:
        for n in (1, 7, 30):
            a.iterate(n)
            st = a.export_state()
            # inactive pairs carry u = 0, so the import restores the activity of every pair with u != 0
            b.import_state(*(st[k].cpu().numpy() for k in ("z", "u_coll", "u_kin", "u_wall")), st["k"])
            a.iterate(1)
            b.iterate(1)
            assert np.array_equal(a.trajectory().cpu().numpy(), b.trajectory().cpu().numpy()), n


@pytest.mark.parametrize("eta", [30, 31, 32, 33, 63, 64])
def test_break_point_counts_around_a_node_warp(eta):
    """One iteration from an oracle iterate, with as many break-points as fill
    a node warp, one fewer, and more than one round of it."""
    prob = twa.Problem.from_instance(workloads.circle_swap(3, eta, 0.15, 0.01, 60 + eta))
    st = par.oracle_state(prob, 4)
    new, info = twa.iterate(prob, st, record_branches=True)
    par.compare(prob, new, info, par.gpu_step(prob, st))
