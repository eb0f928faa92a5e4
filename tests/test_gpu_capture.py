"""Steps captured by the caller between a wall change and the next step that
runs: the first step after the change is launched plainly whether it runs or is
only captured, and a capture does not use up the plain launch of the one that
runs.  The run is that of the same calls without a capture, bit for bit."""
import numpy as np
import pytest

from paper_1604_03478_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_capture_between_wall_and_step(precision):
    import torch
    assert torch.cuda.is_available()
    from paper_1604_03478_gb300 import build, Cavity
    build.build()
    kw = dict(face=0, precision=precision, Ra=1e5, Pr=0.2, Ste=0.6, Ma=0.1, s0=4.3, Tc=-0.1, Tm=0.0, derive=True)
    stream = torch.cuda.Stream()
    out = []
    for capture in (False, True):
        with torch.cuda.stream(stream):
            c = Cavity(34, 14, 12, stream=stream.cuda_stream, **kw)
            c.set_graph_steps(0)
            c.step(4)  # natural layout: the next step is an even one, which reads no wall
            wall = torch.from_numpy((1.0 + inputs.gaussian_field(c.ncols, 0.1, 3)).astype(np.float32)).cuda()
            c.set_hot_wall(wall)
            if capture:
                stream.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    c.step(2)
            c.step(4)
            if capture:
                graph.replay()
            else:
                c.step(2)
            c.step(5)
            out.append(c.get_state())
            c.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
