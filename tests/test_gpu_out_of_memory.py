"""Calls that stage host arrays in device memory when there is none.  A tensor
holds the device's memory but for less than the staging buffers need (all of
both, or the second one only)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KW = dict(face=0, Ra=1e5, Pr=0.1, Ste=0.5, Ma=0.1, s0=20.0, derive=True)
SHAPE = (256, 200, 256)
GB = 1 << 30


def _hold(leave):
    """A tensor over all free device memory but `leave` bytes."""
    import torch
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda")


def _cavity():
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    return Cavity(*SHAPE, **KW)


def test_the_call_after_a_failed_one_succeeds():
    import torch
    from paper_1604_03478_gb300 import _abi, Cavity, LbmError
    c = _cavity()
    held = _hold(int(0.8 * GB))
    with pytest.raises(LbmError) as ei:
        c.get_state()
    assert ei.value.status == _abi.LBM_ENOMEM
    T = c.get()[0]
    assert np.isfinite(T).all()
    with pytest.raises(LbmError) as ei:
        Cavity(*SHAPE, **KW)
    assert ei.value.status == _abi.LBM_ENOMEM
    np.testing.assert_array_equal(c.get()[0], T)
    del held
    torch.cuda.empty_cache()
    c.close()


@pytest.mark.parametrize("leave", [0.8, 1.2])  # f takes 0.93 GiB, g 0.34 GiB
def test_a_failed_upload_changes_nothing(leave):
    """The call gives back what it had allocated, and the cavity steps on like
    one that was never asked."""
    import torch
    from paper_1604_03478_gb300 import _abi, LbmError
    out = []
    for fail in (False, True):
        c = _cavity()
        c.step(7)
        if fail:
            f, g = np.zeros((19, c.N), np.float32), np.zeros((7, c.N), np.float32)
            c.get()
            held = _hold(int(leave * GB))
            free = torch.cuda.mem_get_info()[0]
            for call in (lambda: c.set_state(f, g, np.full(c.ncols, 1.0)), c.get_state):
                with pytest.raises(LbmError) as ei:
                    call()
                assert ei.value.status == _abi.LBM_ENOMEM
                assert torch.cuda.mem_get_info()[0] == free
            del held
            torch.cuda.empty_cache()
        c.step(30)
        out.append(c.get()[:3] + (c.totals()["n_liquid"],))
        c.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
