"""A block shape given by lbm_melt_set_launch after steps in the default layout
takes effect in steps that are replayed from graphs, and so does the default
after it.  Rows of 5 nodes in blocks of 128 threads leave 123 lanes idle where
the default's blocks of 128 consecutive columns leave none: 25 times the
blocks, several waves of them instead of a fraction of one, so several times
the time of a step; 1.5 is the bound."""
import pytest

pytestmark = pytest.mark.gpu


def _us_per_step(c):
    import torch
    best = 1e9
    for _ in range(3):
        c.step(32)
        c.sync()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        c.step(320)
        b.record()
        c.sync()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 320 * 1e3)
    return best


@pytest.mark.parametrize("face", [0, 1])
def test_row_blocks_after_column_blocks(face):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    shape = (5, 200, 400) if face == 0 else (5, 400, 200)
    c = Cavity(*shape, face=face, Ra=1e4, Pr=0.1, Ste=0.1, Ma=0.1, s0=120.0, derive=True)
    columns = _us_per_step(c)
    c.set_launch(128, 1)
    rows = _us_per_step(c)
    c.set_launch(0, 0)
    again = _us_per_step(c)
    print("us a step: columns %.1f, rows %.1f, columns %.1f" % (columns, rows, again))
    assert rows > 1.5 * columns
    assert rows > 1.5 * again
    c.close()
