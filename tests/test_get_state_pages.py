"""REWL.get_state hands the library an array whose pages are there (a device-to-host copy to pages that
are not takes a fault each), by its own writes: the library writes a caller's buffer by the copy alone.
CPU only: the library is a stand-in that looks at the buffer and then fails."""
import ctypes as C
import mmap

import numpy as np
import pytest

import paper_1402_2328_gb300.rewl as R


def _absent_pages(addr, nbytes):
    page = mmap.PAGESIZE
    first = addr // page * page
    n = (addr + nbytes - first + page - 1) // page
    vec = (C.c_ubyte * n)()
    libc = C.CDLL(None, use_errno=True)
    assert libc.mincore(C.c_void_p(first), C.c_size_t(n * page), vec) == 0, C.get_errno()
    return sum(not v & 1 for v in vec)


class _Lib:
    def rewl_get_state(self, handle, name, out, nbytes):
        self.absent = _absent_pages(out.value, nbytes)
        return -2

    def rewl_last_error(self, handle):
        return b"a failing copy"


@pytest.mark.parametrize("field,N,W", [("spins", 9000, 1), ("lng", 1, 3001)])
def test_pages_of_a_large_array_are_present(monkeypatch, field, N, W):
    lib = _Lib()
    monkeypatch.setattr(R, "lib", lambda: lib)
    r = R.REWL.__new__(R.REWL)
    r._lib, r._h, r._owned = lib, C.c_void_p(1), False
    r.h, r.m, r.nw, r.N, r.W = 4, 250, 1000, N, W
    assert r.nw * max(N, 8 * W) > 1 << 20
    with pytest.raises(R.REWLError, match="a failing copy"):
        r.get_state(field)
    assert lib.absent == 0
    r._h = None
