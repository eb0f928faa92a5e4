"""Host arrays that are page-locked in their first pages only.  A kernel must
not be given such an array: the call either copies, with the right values, or
returns the copy's error, and the handle goes on."""
import ctypes as C
import mmap

import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu

PAGE = mmap.PAGESIZE


def _array(n, dtype):
    """n values from the start of a page, with at least two pages."""
    n_bytes = max(n * np.dtype(dtype).itemsize, PAGE + 1)
    m = mmap.mmap(-1, (n_bytes + PAGE - 1) // PAGE * PAGE)
    return np.frombuffer(m, dtype)


def test_part_locked_arrays():
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity, _abi
    build.build()
    L, rt = _abi.load(), torch.cuda.cudart()
    nx = max(128, PAGE // 128)
    kw = dict(face=0, Ra=1e5, Pr=0.1, Ste=1.0, Ma=0.2, s0=3.0, derive=True)
    a, b = Cavity(nx, 12, 80, **kw), Cavity(nx, 12, 80, **kw)
    n = a.ncols
    assert n * 4 > PAGE  # the walls and the fronts reach past the locked page
    wall, S = _array(n, np.float32), _array(n, np.float64)
    wall[:n] = 1.0 + inputs.gaussian_field(n, 0.05, 2)
    lf = C.c_double()
    for arr in (wall, S):
        assert int(rt.cudaHostRegister(arr.ctypes.data, PAGE, 0)) == 0
    try:
        st = L.lbm_melt_set_hot_wall(a._h, C.c_void_p(wall.ctypes.data), 0)
        if st != 0:  # refused: the wall as it was
            a.set_hot_wall(wall[:n].copy())
        b.set_hot_wall(wall[:n].copy())
        for c in (a, b):
            c.step(6)
        st = L.lbm_melt_get_async(a._h, C.c_void_p(S.ctypes.data), C.byref(lf), 0)
        a.sync()
        Sb, lb = b.get(T=False, u=False)[2:]
        if st == 0:
            np.testing.assert_array_equal(S[:n], Sb.ravel())
            assert lf.value == lb
        np.testing.assert_array_equal(a.get()[2], Sb)
    finally:
        for arr in (wall, S):
            rt.cudaHostUnregister(arr.ctypes.data)
    a.close()
    b.close()
