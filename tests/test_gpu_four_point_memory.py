"""Four-point sums on a device without room for the whole scratch.

The device's memory pool is replaced by one of 32 MB (the least there is), so that the first
allocation fails.  The sums must equal those with room.
"""
import ctypes as C

import numpy as np
import pytest

import paper_1710_05155_gb300 as K

pytestmark = pytest.mark.gpu


class PoolProps(C.Structure):
    _fields_ = [("alloc_type", C.c_int), ("handle_types", C.c_int), ("location_type", C.c_int),
                ("location_id", C.c_int), ("security", C.c_void_p), ("max_size", C.c_size_t),
                ("usage", C.c_ushort), ("reserved", C.c_ubyte * 54)]


class SmallPool:
    def __enter__(self):
        self.cuda = C.CDLL("libcuda.so.1")
        self.before, self.pool = C.c_void_p(), C.c_void_p()
        props = PoolProps(1, 0, 1, 0, None, 32 << 20)  # pinned device memory of device 0
        assert self.cuda.cuDeviceGetMemPool(C.byref(self.before), 0) == 0
        assert self.cuda.cuMemPoolCreate(C.byref(self.pool), C.byref(props)) == 0
        assert self.cuda.cuDeviceSetMemPool(0, self.pool) == 0
        return self

    def allocate(self, size):
        at = C.c_uint64(0)
        status = self.cuda.cuMemAllocFromPoolAsync(C.byref(at), C.c_size_t(size), self.pool, None)
        if status == 0:
            assert self.cuda.cuMemFreeAsync(at, None) == 0
        return status

    def __exit__(self, *exc):
        assert self.cuda.cuDeviceSetMemPool(0, self.before) == 0
        assert self.cuda.cuMemPoolDestroy(self.pool) == 0


# slabs in the staging plane; no staging plane; sums without psi
@pytest.mark.parametrize("flags,R,smax,psi", [(0, 64, 100, True), (K.KA_FLAG_GENERIC, 64, 100, True),
                                              (0, 64, 400, False), (K.KA_FLAG_GENERIC, 192, 100, True)])
def test_sums_without_room(flags, R, smax, psi):
    import torch

    with K.Simulation(topo=K.KA_CUBIC, d=3, L=128, m=3, replicas=R, flags=flags) as sim:
        sim.init(5, 0.7)
        sim.sweep(2)
        want = sim.four_point(smax, psi)
        torch.cuda.synchronize()
        with SmallPool() as pool:
            assert pool.allocate(20 << 20) == 0 and pool.allocate(36 << 20) != 0
            got = sim.four_point(smax, psi)
        assert np.array_equal(got[0], want[0])
        assert got[1] is None if not psi else np.array_equal(got[1], want[1])
