"""Single-CTA plans with checkpoint segments longer than one launch runs: the
tape of a segment goes on where the launch before stopped."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,every", [(513, 513), (600, 600), (1100, 1100), (1100, 700), (1030, 515)])
def test_gradients_do_not_depend_on_the_segment_length(K, every):
    import torch
    import paper_1311_4527_gb300 as pk
    inst = workloads.circle_swap(4, 4, 0.05, 0.02, 5)
    gz = torch.randn(4, 5, 2, generator=torch.Generator().manual_seed(K))
    with pk.Planner.from_instance(inst) as pl, pk.Planner.from_instance(inst) as ref:
        ref.profile_start()  # launched kernel by kernel
        out = []
        for p, c in ((pl, every), (pl, 0), (ref, every)):
            p.unroll(K, c)
            out.append([p.trajectory()] + list(p.backward(gz)))
    # the forward pass is the same to the bit; the adjoint's FP32 steps see
    # sums of FP64 atomics in another order, so one may round the other way in
    # each of K iterations: 6e-8 K of the largest entry
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][0], out[2][0])
    for a, b, c in zip(*(o[1:] for o in out)):
        big = float(c.abs().max())
        assert big > 0
        assert float((a - c).abs().max()) <= 6e-8 * K * big and float((b - c).abs().max()) <= 6e-8 * K * big
