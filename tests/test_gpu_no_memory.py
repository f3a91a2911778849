"""Calls that meet a device without free memory: here the device's memory pool
is one of a few MiB, filled up."""
import contextlib
import ctypes

import pytest

from paper_2205_13399_gb300 import inputs

pytestmark = pytest.mark.gpu


class _PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int),
                ("location_type", ctypes.c_int), ("location_id", ctypes.c_int),
                ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


@contextlib.contextmanager
def _full_pool():
    """The device's current pool is a small one with no room left."""
    import torch
    torch.zeros(1, device="cuda")  # the primary context
    cu = ctypes.CDLL("libcuda.so.1")
    old, pool, p = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_uint64()
    props = _PoolProps(alloc_type=1, location_type=1, max_size=4 << 20)  # pinned, on device 0
    assert cu.cuDeviceGetMemPool(ctypes.byref(old), 0) == 0
    if cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) != 0:
        pytest.skip("no pools of a bounded size here")
    taken, total = [], 0
    try:
        for size in (1 << 20, 1 << 14, 512):
            while total < 64 << 20:
                if cu.cuMemAllocFromPoolAsync(ctypes.byref(p), ctypes.c_size_t(size), pool, None):
                    break
                taken.append(p.value)
                total += size
        if total >= 64 << 20:
            pytest.skip("the pool's bound is not kept")
        assert cu.cuDeviceSetMemPool(0, pool) == 0
        yield
    finally:
        cu.cuDeviceSetMemPool(0, old)
        for a in taken:
            cu.cuMemFreeAsync(ctypes.c_uint64(a), None)
        cu.cuCtxSynchronize()
        cu.cuMemPoolDestroy(pool)


def _run(**kw):
    from paper_2205_13399_gb300 import moda
    qi = inputs.uniform_instance(9, index=5, workload="P8")
    inst = moda.Instance(qi.F1, qi.F2, qi.D)
    return inst, moda.anneal(inst, replicas=5, I_max=3000, seed=2, delta0=2e6, deltaf=3e3, xi=0.02,
                             snapshot_every=1000, **kw).wait()


def test_fronts_are_read_without_device_memory():
    _, run = _run()
    want = [run.read_archive(-1), run.read_archive(2), run.read_archive(-1, snapshot=1),
            run.read_archive(3, snapshot=0)]
    with _full_pool():
        got = [run.read_archive(-1), run.read_archive(2), run.read_archive(-1, snapshot=1),
               run.read_archive(3, snapshot=0)]
    assert got == want and len(want[0]) > 1
