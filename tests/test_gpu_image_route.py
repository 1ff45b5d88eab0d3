"""Which images a short exposure adds its pixels to directly: page-locked memory that holds the image whole, in one
allocation or registration, at any offset.  A buffer registered in part, or in two registrations next to each other, is
staged (its pixels past the first one's end have no mapping that the image's first address tells of).  Only the choice is
asked for here; nothing is launched on such memory."""
import ctypes as C
import mmap

import numpy as np
import pytest

from paper_1504_06570_gb300 import phosim as P
from tests import gpu_helpers as G

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

IN_PLACE, STAGED, ADDED = 0, 1, 2
NX = 256                                   # 256 KB of pixels
BYTES = 4 * NX * NX


@pytest.fixture
def route():
    s = P.Scene(G.test_system_scene(chip=NX, atmosphere=False), P.MIXED_DS, early_reject=True)
    f = s.L.phosim_image_route
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_uint64, C.POINTER(C.c_int)]

    def of(address, photons=10):
        out = C.c_int(-1)
        assert f(s.h, address, photons, C.byref(out)) == 0
        return out.value

    yield of
    s.close()


def registered(address, size):
    cudart = torch.cuda.cudart()
    assert int(cudart.cudaHostRegister(address, size, 0)) == 0
    return lambda: cudart.cudaHostUnregister(address)


def test_device_pageable_and_pinned(route):
    device, pageable = torch.zeros(NX * NX, dtype=torch.int32, device="cuda"), torch.zeros(NX * NX, dtype=torch.int32)
    assert route(device.data_ptr()) == IN_PLACE and route(pageable.data_ptr()) == STAGED
    pinned = torch.zeros(3 * NX * NX, dtype=torch.int32).pin_memory()
    direct = route(pinned.data_ptr())
    assert direct in (STAGED, ADDED)       # by whether the GPU adds to host memory natively
    for offset in (0, 4, BYTES, 2 * BYTES):
        assert route(pinned.data_ptr() + offset) == direct
    assert route(pinned.data_ptr(), 10 ** 9) == STAGED


def test_registrations_that_hold_the_image_in_part(route):
    direct = route(torch.zeros(NX * NX, dtype=torch.int32).pin_memory().data_ptr())
    memory = mmap.mmap(-1, 4 * BYTES)
    base = np.frombuffer(memory, np.uint8).ctypes.data
    for pieces in ([(0, BYTES // 2)], [(0, BYTES // 2), (BYTES // 2, BYTES)]):
        undo = [registered(base + at, size) for at, size in pieces]
        assert route(base) == STAGED
        for u in undo:
            u()
    undo = registered(base, 2 * BYTES)
    assert [route(base), route(base + BYTES), route(base + BYTES + 4)] == [direct, direct, STAGED]
    undo()
