"""plan_get_trajectory into a buffer that ends too early is refused, and
nothing behind the buffer is written."""
import contextlib
import ctypes
import mmap

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
SIZE = 1 << 16  # bytes of the short buffer; the trajectory has more


def _runtime():
    import torch  # noqa: F401  (loads the CUDA runtime)
    for line in open("/proc/self/maps"):
        if "libcudart" in line:
            return ctypes.CDLL(line.split()[-1])
    pytest.skip("no shared CUDA runtime in this process")


def _planner():
    import paper_1311_4527_gb300 as pk
    inst = workloads.small_square(600, 16, seed=4)
    assert inst.p * 17 * 8 > SIZE
    return pk, pk.Planner.from_instance(inst)


def _clear(pk, pl):
    """The runtime reports a refused copy once more at the next launch."""
    with contextlib.suppress(pk.PlanError):
        pl.reset()


def test_a_short_device_buffer_is_refused():
    rt = _runtime()
    pk, pl = _planner()
    with pl:
        at = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(at), ctypes.c_size_t(SIZE)) == 0
        status = pk._lib.plan_get_trajectory(pl._h, at, 1)
        assert status != 0
        rt.cudaFree(at)
        _clear(pk, pl)
        assert np.all(np.isfinite(pl.trajectory_host()))  # the plan goes on


def test_a_partly_registered_host_buffer_is_not_written_by_a_kernel():
    rt = _runtime()
    pk, pl = _planner()
    with pl:
        n = pl.p * (pl.eta + 1) * 8
        room = mmap.mmap(-1, 1 << 18)
        host = np.frombuffer(room, np.float32)
        host[:] = -7.0
        at = ctypes.c_void_p(host.ctypes.data)
        assert rt.cudaHostRegister(at, ctypes.c_size_t(SIZE), ctypes.c_uint(0)) == 0
        status = pk._lib.plan_get_trajectory(pl._h, at, 0)
        rt.cudaHostUnregister(at)
        _clear(pk, pl)
        assert np.all(host[n // 4:] == -7.0)
        want = pl.trajectory_host().reshape(-1)  # (a plan that has not moved yet: a reset changes nothing)
        assert status != 0 or np.array_equal(host[:n // 4], want)
