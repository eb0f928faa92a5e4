"""GPU test of the ensemble's launches: a run long enough to replay the
captured launch, with a remainder that is a launch of its own, for both
default launch shapes (a small ensemble and one of more than two items a
block), against single-cavity runs.

Tolerance: the batched kernel may contract multiply-adds differently, half a
unit in the last place (3e-8) a population and step, 150 steps: 5e-6 with all
of them falling the same way."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SMALL = [dict(nx=20, ny=16, nz=12, face=0, Ra=1e5, Pr=0.1, Ste=1.0, Ma=0.2, s0=3.0, derive=True),
         dict(nx=33, ny=14, nz=22, face=1, Ra=3e4, Pr=0.3, Ste=0.5, Ma=0.15, s0=2.5, derive=True)]
LARGE = SMALL + [dict(nx=96, ny=96, nz=96, face=f, Ra=1e5, Pr=0.1, Ste=0.4, Ma=0.1, s0=6.0, derive=True) for f in (0, 1)]


@pytest.mark.parametrize("cases,block", [(SMALL, 256), (LARGE, 128)])
def test_replays_and_remainder(cases, block):
    import torch
    assert torch.cuda.is_available()
    import paper_1604_03478_gb300 as P
    P.build.build()
    ens = P.Ensemble(cases)
    assert ens.info()["block"] == block
    ens.step(150)
    ens.step(1)
    ens.sync()
    for k, c in enumerate(cases):
        c = dict(c)
        one = P.Cavity(c.pop("nx"), c.pop("ny"), c.pop("nz"), **c)
        one.set_node_pairs(0)
        one.step(151)
        a, b = ens.member(k).get_state(), one.get_state()
        for x, y in zip(a, b):
            np.testing.assert_allclose(x, y, atol=5e-6, rtol=0)
        one.close()
    ens.close()
