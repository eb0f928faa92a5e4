"""The routes by which walls, fronts and sums enter and leave a handle:
ordinary host memory (copied), page-locked host memory and device memory (read
and written by the kernels themselves), and device addresses that a kernel
could not use for lack of alignment (copied).  The values are the same bits."""
import ctypes as C

import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu

KW = dict(face=0, Ra=1e5, Pr=0.1, Ste=1.0, Ma=0.2, s0=3.0, derive=True)


def _doubles(n, kind):
    """n doubles of the given kind and their address; kept alive by the tensor."""
    import torch
    if kind == "pageable":
        t = torch.zeros(n, dtype=torch.float64)
        return t, t.data_ptr(), 0
    if kind == "pinned":
        t = torch.zeros(n, dtype=torch.float64).pin_memory()
        return t, t.data_ptr(), 0
    t = torch.zeros(8 * n + 8, dtype=torch.uint8, device="cuda")
    off = 4 if kind == "odd device" else 0
    return t, t.data_ptr() + off, 1


def _values(t, n, kind):
    if kind in ("pageable", "pinned"):
        return t.numpy().copy()
    off = 4 if kind == "odd device" else 0
    return np.frombuffer(t.cpu().numpy().tobytes()[off:off + 8 * n], np.float64)


@pytest.mark.parametrize("nx", [33, 20])
@pytest.mark.parametrize("kind", ["pinned", "device", "odd device"])
def test_same_values_by_every_route(nx, kind):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import Cavity, _abi, build
    build.build()
    L = _abi.load()
    out = {}
    for k in ("pageable", kind):
        c = Cavity(nx, 16, 12, **KW)
        n = c.ncols
        got = []
        for step in range(3):  # natural layout, in flight, natural again
            wall = (1.0 + inputs.gaussian_field(n, 0.02, step)).astype(np.float32)
            w = torch.from_numpy(wall.copy())
            w = w if k == "pageable" else (w.pin_memory() if k == "pinned" else w.cuda())
            assert L.lbm_melt_set_hot_wall(c._h, C.c_void_p(w.data_ptr()), 1 if w.is_cuda else 0) == 0
            c.step(1)
            S, sp, kd = _doubles(n, k)
            lf, lp, _ = _doubles(1, k)
            assert L.lbm_melt_get_async(c._h, C.c_void_p(sp), C.c_void_p(lp), kd) == 0
            c.sync()
            tot, tp, _ = _doubles(7, k)
            assert L.lbm_melt_totals(c._h, C.c_void_p(tp), kd) == 0
            nu, np_, _ = _doubles(n, k)
            mean, mp, _ = _doubles(1, k)
            assert L.lbm_melt_get_nusselt(c._h, C.c_void_p(np_), C.c_void_p(mp), kd) == 0
            S2, s2p, _ = _doubles(n, k)
            l2, l2p, _ = _doubles(1, k)
            assert L.lbm_melt_get(c._h, None, None, C.c_void_p(s2p), C.c_void_p(l2p), kd) == 0
            got += [_values(S, n, k), _values(lf, 1, k), _values(tot, 7, k), _values(nu, n, k), _values(mean, 1, k),
                    _values(S2, n, k), _values(l2, 1, k)]
        # a restart from device fronts, at an aligned and at an odd address
        f, g, s = c.get_state()
        fd, gd = torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()
        S, sp, kd = _doubles(n, k)
        if k in ("device", "odd device"):
            off = 4 if k == "odd device" else 0
            S[off:off + 8 * n] = torch.from_numpy(np.frombuffer(s.tobytes(), np.uint8).copy()).cuda()
        else:
            S, sp, kd = _doubles(n, "device")
            S[:8 * n] = torch.from_numpy(np.frombuffer(s.tobytes(), np.uint8).copy()).cuda()
        assert L.lbm_melt_set_state(c._h, C.c_void_p(fd.data_ptr()), C.c_void_p(gd.data_ptr()), C.c_void_p(sp), 1) == 0
        c.step(2)
        got += list(c.get_state())
        out[k] = got
        c.close()
    for a, b in zip(out["pageable"], out[kind]):
        np.testing.assert_array_equal(a, b)
