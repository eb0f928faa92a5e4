"""The height bound of the stream-collide grid (the running maximum liquid
count, which the front kernel raises in page-locked memory): a handle whose
fronts are replaced by much higher and much lower ones between runs, replayed
from graphs and step by step, against fresh handles given the same state: the
same launches find the same work, so the same bits."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("graph_steps", [16, 0])
def test_fronts_replaced_between_runs(face, graph_steps):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    shape = (37, 90, 11) if face == 0 else (37, 11, 90)
    kw = dict(face=face, Ra=2e4, Pr=0.3, Ste=1.0, Ma=0.15, derive=True)
    a = Cavity(*shape, s0=3.0, **kw)
    a.set_graph_steps(graph_steps)
    a.step(70)
    for s0, steps in ((70.0, 45), (2.0, 101), (40.0, 33)):
        donor = Cavity(*shape, s0=s0, **kw)  # a consistent state with its front at s0
        f, g, s = donor.get_state()
        s = s + inputs.gaussian_field(donor.ncols, 0.2, 3)
        donor.close()
        b = Cavity(*shape, s0=20.0, **kw)
        b.set_graph_steps(0)
        for c in (a, b):
            c.set_state(f, g, s)
            c.step(steps)
        for x, y in zip(a.get_state(), b.get_state()):
            np.testing.assert_array_equal(x, y)
        b.close()
    a.close()
