"""A state uploaded between a recorded run and its backward: the backward
recomputes the recorded run, whose front lies above the uploaded one, so its
buffers and grids follow the run's own height, not the handle's.  The gradient
is that of the same run without the upload, bit for bit, the uploaded state is
left as it was, and the handle steps on from it."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu

STEPS = 23


@pytest.mark.parametrize("face", [0, 1])
@pytest.mark.parametrize("ckpt", [5, STEPS])
def test_backward_after_a_lower_front(face, ckpt):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    shape = (13, 24, 9) if face == 0 else (13, 9, 24)
    kw = dict(face=face, Ra=5e4, Pr=0.3, Ste=0.8, Ma=0.15, derive=True)
    low = Cavity(*shape, s0=1.4, **kw)
    fl, gl, sl = low.get_state()
    got = []
    for upload in (False, True):
        c = Cavity(*shape, s0=9.3, **kw)
        c.tape_forward(STEPS, ckpt)
        if upload:
            c.set_state(fl, gl, sl)
        before = c.get_state()
        got.append(c.tape_backward(inputs.gaussian_field(c.ncols, 1.0, 4)))
        for a, b in zip(before, c.get_state()):
            np.testing.assert_array_equal(a, b)
        if upload:
            c.step(40)
            low.step(40)
            for a, b in zip(c.get_state(), low.get_state()):
                np.testing.assert_array_equal(a, b)
        c.close()
    low.close()
    np.testing.assert_array_equal(got[0][0], got[1][0])
    assert got[0][1] == got[1][1]
