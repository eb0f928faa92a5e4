"""GPU parity of the one-node stream-collide's two kinds of block: the ones of
the first wave, which load before they wait for the front update, and the
later ones.  Grids below, around and above one wave (7 blocks of 128 nodes on
each of the SMs) against the two-nodes-per-thread kernels, which load after
the wait, over steps in which nodes flip after even and odd steps.

Tolerance: the two kernels round FP32 intermediates differently, below 3e-8
a population and step, 26 steps: 1e-6 with all of them falling the same way."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("shape,s0", [((32, 12, 12), 4.0), ((128, 40, 40), 24.0), ((130, 66, 62), 20.0)])
def test_early_and_late_blocks(face, shape, s0):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    kw = dict(face=face, Ra=1e5, Pr=0.2, Ste=0.6, Ma=0.1, s0=s0, derive=True)
    a, b = Cavity(*shape, **kw), Cavity(*shape, **kw)
    a.set_node_pairs(0)
    b.set_node_pairs(1)
    f, g, s = a.get_state()
    s = s0 + inputs.gaussian_field(a.ncols, 0.7, 3 + face)  # fronts over several nodes
    wall = (1.0 + inputs.gaussian_field(a.ncols, 0.05, 5)).astype(np.float32)
    for c in (a, b):
        c.set_state(f, g, s)
        c.set_hot_wall(wall)
        c.step(26)
    (fa, ga, sa), (fb, gb, sb) = a.get_state(), b.get_state()
    assert (np.ceil(sa - 0.5) != np.ceil(s - 0.5)).any()
    np.testing.assert_allclose(sa, sb, atol=1e-6, rtol=0)
    np.testing.assert_allclose(fa, fb, atol=1e-6, rtol=0)
    np.testing.assert_allclose(ga, gb, atol=1e-6, rtol=0)
    a.close()
    b.close()


def _gradient(shape, kw, pairs, steps, spread):
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    c = Cavity(*shape, **kw)
    c.set_node_pairs(pairs)
    if spread:
        f, g, s = c.get_state()
        c.set_state(f, g, s + inputs.gaussian_field(c.ncols, spread, 13))
    c.set_hot_wall((1.0 + inputs.gaussian_field(c.ncols, 0.05, 11)).astype(np.float32))
    S0 = c.get(T=False, u=False, lf=False)[2]
    c.tape_forward(steps, 9)
    S = c.get(T=False, u=False, lf=False)[2]
    dth, par = c.tape_backward(inputs.gaussian_field(c.ncols, 1.0, 12))
    c.close()
    return S0, S, dth, par


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("nx,steps", [(34, 40), (64, 37)])
@pytest.mark.parametrize("spread", [0.0, 0.5])
def test_gradient_with_node_pairs(face, nx, steps, spread):
    """The adjoint's snapshots written by the pair kernels (pairs, pairs split
    by an uneven front, first solid nodes) against those of the one-node
    kernels.  The two forwards differ by FP32 rounding, 1e-6 of T over 40
    steps by the bound above; the gradient is linear in such differences (the
    runs flip the same nodes, as the equal counts say): 1e-4 of its largest
    entry."""
    import torch
    assert torch.cuda.is_available()
    shape = (nx, 20, 14) if face == 0 else (nx, 14, 20)
    kw = dict(face=face, Ra=5e4, Pr=0.3, Ste=0.8, Ma=0.15, s0=3.3, derive=True)
    S0, Sa, da, pa = _gradient(shape, kw, 0, steps, spread)
    _, Sb, db, pb = _gradient(shape, kw, 1, steps, spread)
    np.testing.assert_array_equal(np.ceil(Sa - 0.5), np.ceil(Sb - 0.5))
    if spread:
        assert (np.ceil(Sa - 0.5) != np.ceil(S0 - 0.5)).any()  # nodes flipped
    assert np.abs(da - db).max() <= 1e-4 * np.abs(da).max()
    for k in pa:
        assert abs(pa[k] - pb[k]) <= 1e-4 * max(abs(pa[k]), 1e-12)


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("nx,pairs,solid", [(1, 0, 0), (5, 0, 0), (33, 0, 0), (71, 0, 1), (130, 0, 0), (6, 1, 0),
                                            (38, 1, 0), (70, 1, 1), (140, 1, 0)])
@pytest.mark.parametrize("precision", [0, 1])
def test_columns_in_a_line(face, nx, pairs, solid, precision):
    """Stream-collide blocks of consecutive columns (rows that leave lanes
    idle) against blocks of rows: the same threads do the same arithmetic, so
    the states are the same bits."""
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    shape = (nx, 11, 7) if face == 0 else (nx, 7, 11)
    kw = dict(face=face, precision=precision, Ra=5e4, Pr=0.3, Ste=0.8, Ma=0.15, s0=4.2, derive=True)
    if solid:
        kw.update(solid=1, ks_kl=0.7, Tc=-0.2)
    out = []
    for rows in (False, True):
        c = Cavity(*shape, **kw)
        c.set_node_pairs(pairs)
        if rows:
            c.set_launch(32, 2)
        f, g, s = c.get_state()
        c.set_state(f, g, s + inputs.uniform(c.ncols, -1.2, 1.2, 17))
        c.step(19)
        out.append(c.get_state())
        c.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
