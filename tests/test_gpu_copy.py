"""plan_get_trajectory into each kind of buffer (device, off a 16-byte
boundary, pinned and pageable host memory) gives the same break-points and
writes nothing else, at even and odd counts of them."""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,eta", [(1, 2), (3, 2), (5, 3), (130, 16)])
def test_every_destination_gets_the_same(p, eta):
    import torch
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(p, eta, seed=7)
    n = p * (eta + 1) * 2
    with pk.Planner.from_instance(inst) as pl:
        pl.iterate(3)
        want = pl.export_state()["z"].cpu().numpy().reshape(-1)
        for off in (0, 1, 2, 4):
            dev = torch.full((n + 16,), -7.0, device=pl.device)
            pin = torch.full((n + 16,), -7.0).pin_memory()
            page = np.full(n + 16, -7.0, np.float32)
            for at, on_device in ((dev.data_ptr(), 1), (pin.data_ptr(), 0), (page.ctypes.data, 0)):
                assert pk._lib.plan_get_trajectory(pl._h, ctypes.c_void_p(at + 4 * off), on_device) == 0
            torch.cuda.synchronize()
            for got in (dev.cpu().numpy(), pin.numpy(), page):
                assert np.array_equal(got[off:off + n], want)
                assert np.all(got[:off] == -7.0) and np.all(got[off + n:] == -7.0)
