"""F1 of covers where there is no room for the table of ranges: the reference
memberships are searched instead, and the result is the same.  The room is
bounded on the host side: the process allocates from a memory pool of its own
with a maximum size, which holds everything the call needs except the table
(8 bytes per id)."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOM = 96 << 20


class Location(C.Structure):
    _fields_ = [("type", C.c_int), ("id", C.c_int)]


class PoolProps(C.Structure):   # CUmemPoolProps
    _fields_ = [("allocType", C.c_int), ("handleTypes", C.c_int), ("location", Location),
                ("win32SecurityAttributes", C.c_void_p), ("maxSize", C.c_size_t), ("usage", C.c_ushort),
                ("reserved", C.c_ubyte * 54)]


@pytest.fixture
def small_pool():
    import torch
    torch.cuda.init()
    torch.zeros(1, device="cuda")   # the primary context
    dev = torch.cuda.current_device()
    cu = C.CDLL("libcuda.so.1")
    pool, old = C.c_void_p(), C.c_void_p()
    props = PoolProps(allocType=1, location=Location(1, dev), maxSize=ROOM)   # pinned, on this device
    assert cu.cuDeviceGetMemPool(C.byref(old), dev) == 0
    if cu.cuMemPoolCreate(C.byref(pool), C.byref(props)) != 0:
        pytest.skip("no memory pools with a maximum size")
    assert cu.cuDeviceSetMemPool(dev, pool) == 0
    yield
    assert cu.cuDeviceSetMemPool(dev, old) == 0
    cu.cuMemPoolDestroy(pool)


def covers():
    rng = np.random.default_rng(5)
    top = 15_500_000
    ref = [np.unique(rng.integers(0, top, 1000)).astype(np.int32) for _ in range(1000)]
    det = [np.unique(np.concatenate([rng.choice(ref[int(i)], 200) for i in rng.integers(0, 1000, 3)])) for _ in range(50)]
    assert 8 * top > ROOM and top < 16 * sum(len(c) for c in ref)
    return det, ref


def test_f1_without_room_for_the_table(small_pool):
    import oracle
    from paper_2210_03211_gb300 import lazyfox
    det, ref = covers()
    want, best = oracle.cover_f1(det, ref)
    got, gbest = lazyfox.cover_f1(det, ref)
    assert got == want and np.array_equal(gbest, best)
