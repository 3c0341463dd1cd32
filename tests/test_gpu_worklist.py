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


@pytest.mark.parametrize("p,eta,iters", [(2047, 21, 40), (2880, 11, 20)])
def test_sorted_tiles_give_the_dense_iterates(p, eta, iters):
    """Plans large enough for sorted tiles, over several sorts, with new fixed
    ends in between (boxes widened, not sorted anew) and an imported state."""
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(p, eta, seed=90 + p)
    moved = (0.98 * inst.start + 0.02 * inst.start.mean(0), inst.goal)
    shrunk = 0.9 * inst.radius  # so that the moved starts stay clear of one another
    out = []
    for flags in (0, pk.PLAN_DENSE_STATE):
        with pk.Planner.from_instance(inst, flags=flags) as pl:
            pl.set_params(radius=shrunk)
            zs = []
            for n in (3, iters - 3):
                pl.iterate(n)
                zs.append((pl.trajectory().cpu().numpy(), pl.info()["active_coll"]))
            pl.set_endpoints(*moved)
            pl.iterate(9)
            zs.append((pl.trajectory().cpu().numpy(), pl.info()["active_coll"]))
        out.append(zs)
    for (zg, ag), (zd, ad) in zip(*out):
        assert np.array_equal(zg, zd) and ag == ad


@pytest.mark.parametrize("eta", [30, 31, 32, 33, 63, 64])
def test_break_point_counts_around_a_node_warp(eta):
    """One iteration from an oracle iterate, with as many break-points as fill
    a node warp, one fewer, and more than one round of it."""
    prob = twa.Problem.from_instance(workloads.circle_swap(3, eta, 0.15, 0.01, 60 + eta))
    st = par.oracle_state(prob, 4)
    new, info = twa.iterate(prob, st, record_branches=True)
    par.compare(prob, new, info, par.gpu_step(prob, st))


@pytest.mark.parametrize("p,eta", [(2, 1), (5, 3), (20, 8), (28, 4), (29, 4), (16, 8)])
def test_single_cta_runs_equal_iterations_one_kernel_at_a_time(p, eta):
    """Problems on both sides of the single-CTA rule: runs of iterations
    against the same iterations launched kernel by kernel (profiling), with
    odd run lengths, the feasibility mode and walls."""
    import paper_1311_4527_gb300 as pk
    for inst, kw in ((workloads.circle_swap(p, eta, 0.04, 0.005, 3), {}),
                     (workloads.circle_swap(p, eta, 0.04, 0.005, 3), {"energy": False}),
                     (workloads.small_square(p, eta, seed=p), {"vmax": 0.4})):
        out = []
        for single in (True, False):
            with pk.Planner.from_instance(inst, **kw) as pl:
                if not single:
                    pl.profile_start()
                zs = []
                for n in (1, 1, 6, 33):
                    pl.iterate(n)
                    zs.append(pl.trajectory().cpu().numpy())
                out.append(zs + [pl.iterate(2, residual=True)])
        for a, b in zip(*out):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("p,eta,K,C", [(4, 4, 23, 5), (40, 4, 23, 5), (40, 4, 24, 6), (33, 2, 7, 7)])
def test_backward_by_graph_and_by_one_cta_match_single_launches(p, eta, K, C):
    """The captured segments (odd and even lengths, the first one and the
    rest, called again with another loss) and the single-CTA form against the
    same steps launched one by one: equal up to the order of FP64 atomics."""
    import torch
    import paper_1311_4527_gb300 as pk
    inst = workloads.circle_swap(p, eta, 0.03, 0.005, 7)
    gen = torch.Generator().manual_seed(3)
    losses = [torch.randn(p, eta + 1, 2, generator=gen) for _ in range(2)]
    with pk.Planner.from_instance(inst) as pl, pk.Planner.from_instance(inst) as ref:
        pl.unroll(3, 2)  # another layout first
        pl.backward(losses[0])
        ref.profile_start()
        for g in losses:
            pl.unroll(K, C)
            ref.unroll(K, C)
            assert torch.equal(pl.trajectory(), ref.trajectory())
            for a, b in zip(pl.backward(g), ref.backward(g)):
                assert torch.allclose(a, b, rtol=1e-5, atol=1e-6 * float(b.abs().max()))


@pytest.mark.parametrize("p,eta", [(33, 3), (200, 8), (384, 17)])
def test_dense_blocks_of_each_size_equal_the_batch(p, eta):
    """A single plan's blocks of pairs (16, 8 and 4 warps, minimizers run by
    the block) against the batch's (minimizers from the members' worklists)."""
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(p, eta, seed=140 + p)
    for flags in (pk.PLAN_DENSE_STATE, pk.PLAN_U_KEEP, pk.PLAN_ADMM):
        with pk.Planner.from_instance(inst, flags=flags) as a, pk.PlannerBatch([inst], flags=flags) as b:
            for n in (1, 2, 9):
                a.iterate(n)
                b.iterate(n)
                assert np.array_equal(a.trajectory().cpu().numpy(), b.trajectory(0).cpu().numpy()), (flags, n)
            assert a.info()["active_coll"] > 0


@pytest.mark.parametrize("p,eta", [(1, 12), (28, 8), (29, 8), (8, 12), (8, 13), (8, 3), (40, 2)])
def test_single_cta_rule_edges(p, eta):
    """Up to one and a half rounds of the CTA's warps and both pair limits."""
    test_single_cta_runs_equal_iterations_one_kernel_at_a_time(p, eta)
