"""The totals are FP64 sums: their error stays within FP64 rounding where a
value a few bits below the running sum's 48th is added again and again (a sum
held as a pair of FP32 values drops it).

Tolerance: a thread adds at most 8 nodes, a block's tree has 8 levels, the last
block adds at most two partials a thread and has 8 levels: 26 roundings of
2^-53 of the sum.  The eight nodes of a column are 1, just under 2^-24, and six
of 0.9 2^-49: without the six the sum is 86 times 2^-53 too low."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("face", [0, 1])
def test_sum_of_temperatures(face):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    shape = (32, 16, 12) if face == 0 else (32, 12, 16)
    c = Cavity(*shape, face=face, Ra=1e4, Pr=0.1, Ste=0.1, Ma=0.1, s0=8.2, derive=True)
    f, g, s = c.get_state()
    col = np.zeros(16, np.float32)
    col[:8] = [1.0, (2 ** 24 - 1) * 2.0 ** -48] + [0.9 * 2.0 ** -49] * 6
    T = np.zeros(c.shape, np.float32)
    T[...] = col[None, :, None] if face == 0 else col[:, None, None]
    g[:] = 0.0
    g[0] = T.ravel()
    c.set_state(f, g, np.full(c.ncols, 8.2))
    np.testing.assert_array_equal(c.get()[0], T)
    exact = math.fsum(T.ravel().tolist())
    t = c.totals()
    assert t["n_liquid"] == 8 * c.ncols
    assert abs(t["sum_T_minus_Tm"] - exact) <= 26 * 2.0 ** -53 * exact
    c.close()
