"""The local planner's epoch forms its reference targets and its new positions
with one rounding per coordinate (a fused multiply-add), so that an epoch does
not depend on how the library was compiled."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_targets_and_positions_are_rounded_once():
    import paper_1311_4527_gb300 as pk
    f = np.float32
    rng = np.random.default_rng(2)
    p, step, advance = 200, 0.13, 0.3
    a = np.arange(p) * (2 * np.pi / p)
    x0 = (20 * np.stack([np.cos(a), np.sin(a)], 1) + rng.uniform(-0.01, 0.01, (p, 2))).astype(f)
    dest = (x0 + rng.uniform(0.5, 2.0, (p, 2))).astype(f)
    with pk.Planner.velocity_obstacle(x0, dest, np.full(p, 0.05), np.ones(p), step, rho0=30.0, alpha=0.5,
                                      tol=1e-9, max_iter=3, check_every=3) as pl:
        pl.vo_epoch(advance)
        z = pl.trajectory().cpu().numpy()
        new, ref = (np.asarray(v.cpu() if hasattr(v, "cpu") else v) for v in pl.endpoints())
    once = lambda s, d, at: (f(s).astype(np.float64) * d.astype(np.float64) + at.astype(np.float64)).astype(f)
    assert np.array_equal(new, once(advance, z[:, 1] - x0, x0))
    d = dest - x0
    # the length may be a unit in the last place either way: one of the three scales explains a target
    L = np.hypot(d[:, 0], d[:, 1])
    fits = [np.all(ref == once((f(step) / l)[:, None], d, x0), 1)
            for l in (L, np.nextafter(L, f(0)), np.nextafter(L, f(9)))]
    assert np.all(fits[0] | fits[1] | fits[2])
