"""Host output buffers made resident before a copy keep their contents: a call
that fails before its copy leaves the caller's array as it was.

The function under test is internal (lqcd::prefault_host), called by its
exported C++ name; it makes no CUDA call.  Buffers: fresh pages (resident
nowhere), resident ones, resident only at the places that are looked at or
only elsewhere, odd start addresses, and sizes around the 4 MB limit and the
shares of the threads."""
import ctypes
import mmap

import numpy as np
import pytest

MB = 1 << 20
PAGE = mmap.PAGESIZE


@pytest.fixture(scope="module")
def prefault():
    from paper_1701_00426_gb300 import build
    f = ctypes.CDLL(build.build())._ZN4lqcd13prefault_hostEPvm
    f.argtypes = [ctypes.c_void_p, ctypes.c_size_t]
    f.restype = None
    return f


@pytest.mark.parametrize("size", [1, 4 * MB - 1, 4 * MB, 4 * MB + 1, 9 * MB + 17, 33 * MB + PAGE - 1])
@pytest.mark.parametrize("offset", [0, 1, PAGE - 1])
@pytest.mark.parametrize("filled", ["all", "first half", "every 40th page"])
def test_contents_stay(prefault, size, offset, filled):
    m = mmap.mmap(-1, size + 2 * PAGE)
    whole = np.frombuffer(m, dtype=np.uint8)
    pages = range(0, whole.size, PAGE)
    if filled == "all":
        whole[:] = np.random.default_rng(size + offset).integers(1, 256, whole.size, dtype=np.uint8)
    else:
        for k, p in enumerate(pages):
            if (filled == "first half" and p < whole.size // 2) or (filled != "first half" and k % 40 == 0):
                whole[p:p + PAGE] = 1 + k % 255
    want = whole.copy() if filled == "all" else None
    prefault(whole.ctypes.data + offset, size)
    if want is not None:
        assert np.array_equal(whole, want)
        return
    for k, p in enumerate(pages):
        lit = (filled == "first half" and p < whole.size // 2) or (filled != "first half" and k % 40 == 0)
        assert (whole[p:p + PAGE] == (1 + k % 255 if lit else 0)).all()
