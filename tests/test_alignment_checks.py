"""Device pointers that the kernels' accesses do not allow are refused on the host, before any CUDA
call (fake addresses: nothing here touches a device)."""
import ctypes as C

import numpy as np
import pytest

BASE = 1 << 40
BYTES = {0: 8, 1: 4, 2: 2, 3: 2, 4: 1, 5: 4, 6: 2}


@pytest.fixture(scope="module")
def L():
    import paper_2009_12101_gb300 as cb
    cb.ensure_built()
    return cb.lib()


@pytest.mark.parametrize("fmt", range(7))
def test_misaligned_pointers_are_refused(L, fmt):
    n, ld, nc = 4096, 4096, 2
    h = np.zeros(8)
    hp = C.c_void_p(h.ctypes.data)
    for off in (1, BYTES[fmt], 4, 8):
        if off % 16 == 0:
            continue
        for arith in (0, 1):
            assert L.cbg_basis_dot(fmt, arith, n, nc, BASE + off, ld, hp, BASE, hp, None) == -1
            assert L.cbg_basis_axpy(fmt, arith, n, nc, BASE + off, ld, hp, hp, BASE, None) == -1
            assert L.cbg_basis_dot_noalloc(fmt, arith, n, nc, BASE + off, ld, hp, BASE, hp, None) == -1
    assert L.cbg_basis_dot(fmt, 1, n, nc, BASE, ld, hp, BASE + 8, hp, None) == -1
    assert L.cbg_basis_dot(fmt, 0, n, nc, BASE, ld, hp, BASE + 4, hp, None) == -1
    assert L.cbg_basis_axpy(fmt, 0, n, nc, BASE, ld, hp, hp, BASE + 4, None) == -1
    assert L.cbg_basis_dot_noalloc(fmt, 0, n, nc, BASE, ld, hp, BASE + 8, hp, None) == -1
    big = 1 << 40
    if BYTES[fmt] > 1:
        assert L.cbg_basis_dot_multi_path(fmt, n, nc, BASE + 1, ld, BASE, 2, BASE, n, BASE, BASE, big, None, 1) == -1
    for scales, w, out in ((BASE + 4, BASE, BASE), (BASE, BASE + 4, BASE), (BASE, BASE, BASE + 4)):
        assert L.cbg_basis_dot_multi_path(fmt, n, nc, BASE, ld, scales, 2, w, n, out, BASE, big, None, 1) == -1
