"""Mapping the pages of an output buffer before a device-to-host copy: a buffer whose
pages are there costs next to nothing, a fresh one is mapped and keeps its bytes."""
import ctypes as C
import mmap
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def prefault():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_04565_gb300 import lsm
    torch.zeros(1, device="cuda")
    f = C.CDLL(lsm.LIB_PATH)._ZN3lsm8prefaultEPvm
    f.restype, f.argtypes = None, [C.c_void_p, C.c_size_t]
    return f


def _resident(buf, size):
    page = mmap.PAGESIZE
    addr = C.addressof(C.c_char.from_buffer(buf))
    vec = (C.c_ubyte * (size // page))()
    assert C.CDLL(None).mincore(C.c_void_p(addr), C.c_size_t(size), vec) == 0
    return np.frombuffer(vec, np.uint8) & 1


@pytest.mark.parametrize("size,bound", [(8 << 10, 4e-6), (1 << 20, 6e-6), (24 << 20, 20e-6)])
def test_mapped_buffer_costs_little(prefault, size, bound):
    """Far below the copy of such a buffer (9, 15 and 130 us). It was 11 us and, with
    its threads, 90 us."""
    buf = np.ones(size, np.uint8)
    best = 1.0
    for _ in range(200):
        t = time.perf_counter()
        prefault(buf.ctypes.data, size)
        best = min(best, time.perf_counter() - t)
    assert best < bound
    assert (buf == 1).all()


@pytest.mark.parametrize("size,touched", [(576 << 10, 0), (3 << 20, 0), (46 << 20, 9), (320 << 20, 4500)])
def test_fresh_buffer_is_mapped(prefault, size, touched):
    pages = size // mmap.PAGESIZE
    buf = mmap.mmap(-1, size, flags=mmap.MAP_PRIVATE | mmap.MAP_ANONYMOUS)
    buf[:touched * mmap.PAGESIZE] = b"\x07" * (touched * mmap.PAGESIZE)
    assert _resident(buf, size).sum() < pages
    prefault(C.addressof(C.c_char.from_buffer(buf)) + 5, size - 9)
    assert _resident(buf, size).all()
    a = np.frombuffer(buf, np.uint8)
    assert (a[:touched * mmap.PAGESIZE] == 7).all() and not a[touched * mmap.PAGESIZE:].any()


def test_odd_arguments(prefault):
    prefault(None, 100)
    prefault(np.ones(4).ctypes.data, 0)
    prefault(C.c_void_p(1 << 45), 1 << 20)  # nothing there
