"""Gradients of one handle with few and with many checkpoints, in turn, where
the device has room for either run's buffers but not for both runs': buffers
kept from the run before must not stand in the way.  A tensor holds the rest of
the device's memory."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu

GB = 1 << 30
STEPS = 40


def _hold(leave):
    import torch
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda")


def _setup():
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    c = Cavity(64, 64, 64, face=0, Ra=5e4, Pr=0.3, Ste=0.8, Ma=0.15, s0=50.0, derive=True)
    return c, c.get_state(), inputs.gaussian_field(c.ncols, 1.0, 6)


@pytest.mark.parametrize("order", [(1, STEPS), (STEPS, 1)])
def test_buffers_of_the_run_before(order):
    """1: 40 checkpoints (1.0 GiB) and snapshots of two levels; 40: one
    checkpoint and snapshots of 41 levels (0.85 GiB, twice where there is
    room)."""
    import torch
    c, start, seed = _setup()

    def gradient(every):
        c.set_state(*start)
        c.tape_forward(STEPS, every)
        return c.tape_backward(seed)

    want = [gradient(every) for every in order]
    c.tape_clear()
    c.set_state(*start)
    held = _hold(int(1.5 * GB))
    for every, w in zip(order, want):
        got = gradient(every)
        np.testing.assert_array_equal(got[0], w[0])
        assert got[1] == w[1]
    del held
    torch.cuda.empty_cache()
    c.close()


def test_backward_after_one_without_room():
    """A backward without room for its buffers says so and keeps the recorded
    run: asked again with room, it gives the gradient."""
    import torch
    from paper_1604_03478_gb300 import _abi, LbmError
    c, start, seed = _setup()
    c.tape_forward(STEPS, STEPS)
    want = c.tape_backward(seed)
    c.tape_clear()
    c.set_state(*start)
    c.tape_forward(STEPS, STEPS)
    held = _hold(int(0.5 * GB))  # the snapshots take 0.85 GiB
    with pytest.raises(LbmError) as ei:
        c.tape_backward(seed)
    assert ei.value.status == _abi.LBM_ENOMEM
    del held
    torch.cuda.empty_cache()
    got = c.tape_backward(seed)
    np.testing.assert_array_equal(got[0], want[0])
    assert got[1] == want[1]
    c.close()
