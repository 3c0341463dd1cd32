"""The FP32 minimizers depend on their weights' ratio only: with both weights
scaled by a power of two, over the range that rho0 may have, the outputs are
the same to the bit.  CPU only (needs nvcc, which builds the harness)."""
import numpy as np
import pytest

from test_minimizers_host import H, _capsule, _disk  # noqa: F401


@pytest.mark.parametrize("w", [2.0 ** -80, 2.0 ** -66, 2.0 ** 66, 2.0 ** 90])
def test_minimizers_do_not_depend_on_the_size_of_the_weights(H, w):  # noqa: F811
    rng = np.random.default_rng(8)
    for _ in range(3000):
        a, b, c0, c1 = rng.normal(0, 1.0, (4, 2))
        assert np.array_equal(_disk(H, a, b, w, w, 0.7), _disk(H, a, b, 1.0, 1.0, 0.7))
        assert np.array_equal(_capsule(H, a, b, w, w, c0, c1, 0.4), _capsule(H, a, b, 1.0, 1.0, c0, c1, 0.4))
