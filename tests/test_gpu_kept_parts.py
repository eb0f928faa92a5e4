"""lbm_melt_set_state with f or g (or both) left out, between an even and an odd
step: the part that is kept is the state's own, the other the given one, as in
the natural layout after the read-out of the whole state."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("solid", [0, 1])
@pytest.mark.parametrize("given", ["", "f", "g", "fg"])
def test_kept_parts_in_flight(face, solid, given):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    shape = (18, 14, 11) if face == 0 else (18, 11, 14)
    kw = dict(face=face, Ra=5e4, Pr=0.3, Ste=0.8, Ma=0.15, s0=4.2, derive=True)
    if solid:
        kw.update(solid=1, ks_kl=0.7, Tc=-0.2)
    a, b = Cavity(*shape, **kw), Cavity(*shape, **kw)
    for c in (a, b):
        c.step(9)  # in flight
    f, g, s = a.get_state()
    new = dict(f=f * (1.0 + inputs.uniform(f.shape, -1e-3, 1e-3, 1)).astype(np.float32),
               g=g * (1.0 + inputs.uniform(g.shape, -1e-3, 1e-3, 2)).astype(np.float32))
    a.set_state(f=new["f"] if "f" in given else None, g=new["g"] if "g" in given else None)
    b.set_state(f=new["f"] if "f" in given else f, g=new["g"] if "g" in given else g)
    for c in (a, b):
        c.step(5)
    for x, y in zip(a.get_state(), b.get_state()):
        np.testing.assert_array_equal(x, y)
    a.close()
    b.close()
