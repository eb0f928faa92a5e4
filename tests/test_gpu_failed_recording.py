"""A recorded forward that fails part-way leaves no recorded run.  It is made to
fail on the host: within a capture, the events by which the host follows the
liquid's height are captured too, and waiting for one is an error.  In a process
of its own, which ends with the broken capture."""
import os
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

CHILD = """
import numpy as np, torch
from paper_1604_03478_gb300 import _abi, build, Cavity, LbmError
build.build()
stream = torch.cuda.Stream()
with torch.cuda.stream(stream):
    c = Cavity(18, 14, 12, face=0, Ra=5e4, Pr=0.3, Ste=0.8, Ma=0.15, s0=4.2, derive=True, stream=stream.cuda_stream)
    c.set_graph_steps(0)
    c.tape_forward(60, 6)  # the buffers
    c.tape_backward(np.ones(c.ncols))
    failed = None
    try:
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=stream, capture_error_mode="relaxed"):
            try:
                c.tape_forward(60, 6)
            except LbmError as e:
                failed = e.status
    except RuntimeError:  # the capture does not survive
        pass
    assert failed == _abi.LBM_ECUDA, failed
    try:
        c.tape_backward(np.ones(c.ncols))
        print("accepted")
    except LbmError as e:
        print("status", e.status == _abi.LBM_EINVAL)
import os, sys
sys.stdout.flush()
os._exit(0)
"""


def test_no_run_after_a_failed_recording():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.stdout.strip() == "status True", r.stdout + r.stderr
