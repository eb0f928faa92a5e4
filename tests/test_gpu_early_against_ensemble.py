"""The stream-collide kernels that load before they wait for the front update
(one and two nodes per thread, grids below, around and above one wave of
blocks), and the two-nodes-per-thread kernels above 160^3 nodes, which do not,
against the ensemble's kernel: it loads behind a grid barrier only, so a value
read too early shows.  Wavy fronts, so that nodes flip after even and odd steps,
and a wall changed in flight.

Tolerance: the kernels round FP32 intermediates differently, below 3e-8 a
population and step, 27 steps: 1e-6 with all of them falling the same way."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("shape,s0", [((32, 12, 12), 4.0), ((128, 40, 40), 24.0), ((130, 66, 62), 20.0),
                                      ((256, 126, 132), 60.0)])
def test_early_loads_against_the_ensemble(face, shape, s0):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity, Ensemble
    build.build()
    kw = dict(face=face, Ra=1e5, Pr=0.2, Ste=0.6, Ma=0.1, s0=s0, derive=True)
    ens = Ensemble([dict(nx=shape[0], ny=shape[1], nz=shape[2], **kw)])
    large = np.prod(shape) > 160 ** 3
    cavs = [ens.member(0)] + [Cavity(*shape, **kw) for _ in range(2)]
    cavs[1].set_node_pairs(0)
    cavs[2].set_node_pairs(-1 if large else 1)
    f, g, s = cavs[1].get_state()
    s = s0 + inputs.gaussian_field(cavs[1].ncols, 0.7, 3 + face)
    walls = [(1.0 + inputs.gaussian_field(cavs[1].ncols, 0.05, k)).astype(np.float32) for k in (5, 6)]
    for c in cavs:
        step = ens.step if c is cavs[0] else c.step
        c.set_state(f, g, s)
        c.set_hot_wall(walls[0])
        step(9)
        c.set_hot_wall(walls[1])
        step(18)
    ens.sync()
    want = cavs[0].get_state()
    assert (np.ceil(want[2] - 0.5) != np.ceil(s - 0.5)).any()
    for c in cavs[1:]:
        for a, b in zip(c.get_state(), want):
            np.testing.assert_allclose(a, b, atol=1e-6, rtol=0)
        c.close()
    ens.close()
