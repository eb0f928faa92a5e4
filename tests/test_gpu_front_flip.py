"""GPU parity of the merged front update and phase flip: fronts a hair from
node centres, with liquid warmer than Tm in some columns and colder in others,
so that neighbouring columns melt and refreeze nodes in the same step, after
even steps (values in flight) and odd ones; every reader of the state between
steps (distributions, fields, totals) against the FP64 oracle.

Tolerance: an FP32 step rounds each population (below 1/2 in magnitude) in
about thirty operations of half a unit in the last place, 3e-8 each relative:
below 1e-6 a step when all fall the same way, 4e-6 over the four steps."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu

W19 = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
W7 = np.array([1 / 4] + [1 / 8] * 6)
TOL = 4e-6


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    return Cavity


def _mixed_state(o, seed):
    """Fronts 0.004 to 0.02 below (warm columns) or above (cold columns) a
    node centre; T linear from +-0.4 at the wall to Tm at the front."""
    nz, ny, nx = o.shape
    k = np.floor(inputs.uniform(o.ncols, 2.0, 7.0, seed)) + 0.5
    warm = inputs.uniform(o.ncols, 0.0, 1.0, seed + 1) < 0.5
    s = np.where(warm, k - inputs.uniform(o.ncols, 0.004, 0.02, seed + 2), k + inputs.uniform(o.ncols, 0.004, 0.02, seed + 2))
    Z, Y, X = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    col = (Z * nx + X) if o.face == 0 else (Y * nx + X)
    a = (Y if o.face == 0 else Z) + 0.5
    sc, sign = s[col], np.where(warm, 0.4, -0.4)[col]
    liq = (a < sc).reshape(-1)
    T = np.where(a < sc, sign * (1.0 - a / sc), 0.0).reshape(-1)
    f = inputs.noisy(np.tile(W19[:, None], (1, o.N)), 2e-3, seed + 3)
    f[:, ~liq] = 0.0
    g = W7[:, None] * T[None, :]
    return f.astype(np.float32), g.astype(np.float32), s


@pytest.mark.parametrize("face,shape,pairs", [(0, (33, 10, 5), 0), (1, (33, 5, 10), 0), (0, (34, 10, 5), 1),
                                              (1, (2, 3, 10), 1), (0, (1, 10, 1), 0)])
def test_melting_and_refreezing_neighbours(lib, orc, face, shape, pairs):
    kw = dict(face=face, Ra=2e3, Ste=0.5, s_nu=1.3, s_alpha=1.2)
    gpu, o = lib(*shape, **kw), orc.Oracle(*shape, **kw)
    gpu.set_node_pairs(pairs)
    f, g, s = _mixed_state(o, 31 + face)
    # the wall follows the columns' sign, or their nodes next to it turn
    wall = np.where(g.sum(0).reshape(o.shape)[(slice(None), 0) if face == 0 else 0].ravel() < 0, -0.4, 0.4)
    o.set_hot_wall(wall)
    gpu.set_hot_wall(wall.astype(np.float32))
    o.set_state(f.astype(np.float64), g.astype(np.float64), s)
    gpu.set_state(f, g, s)
    changed = 0
    for n in range(4):
        before = np.ceil(o.get_state()[2] - 0.5)
        gpu.step(1)
        o.step(1)
        fg, gg, sg = gpu.get_state()
        fo, go, so = o.get_state()
        d = np.ceil(so - 0.5) - before
        changed += int((d > 0).any()) + int((d < 0).any())
        liq = fo.any(axis=0)
        np.testing.assert_allclose(sg, so, atol=TOL, rtol=0)
        np.testing.assert_allclose(fg, fo, atol=TOL, rtol=0)
        np.testing.assert_allclose(gg[:, liq], go[:, liq], atol=TOL, rtol=0)
        Tg, ug, _, _ = gpu.get()
        To, uo, _, _ = o.get()
        np.testing.assert_allclose(Tg, To, atol=7 * TOL, rtol=0)
        np.testing.assert_allclose(ug, uo, atol=10 * TOL, rtol=0)
        t = gpu.totals()
        assert t["n_liquid"] == int(liq.sum())
        assert abs(t["sum_rho_minus_1"] - float((fo.sum(0) - 1.0)[liq].sum())) <= 19 * TOL * max(1, liq.sum())
    if shape[0] > 1:
        assert changed >= 2  # nodes melted and nodes refroze
    gpu.close()
