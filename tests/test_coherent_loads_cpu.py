"""What the front update writes (liquid counts js, bounds nb, ghost populations
gpost and spost) is never read by the stream-collide through the non-coherent
path: its early blocks are resident while the front update still writes, and
the ensemble's kernel writes these arrays itself.  That path is taken by __ldg
and allowed by a const __restrict__ kernel parameter; both are looked for in
the source, above the front update's own section."""
import os
import re

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_1604_03478_gb300", "csrc")


@pytest.mark.parametrize("name", ["kernels.cuh", "k_cond.cu", "ensemble_kernel.cuh", "lbm_core.cuh"])
def test_front_arrays_are_read_coherently(name):
    with open(os.path.join(CSRC, name)) as fh:
        text = fh.read()
    if name == "kernels.cuh":
        text, rest = text.split("front (Eq. 6)\n// One thread per column")
        assert "k_front" in rest
    text = re.sub(r"//[^\n]*", "", text)
    arrays = r"(js|js_old|nb|nb_old|gpost|spost|gbuf)\b"
    text = text.replace("FIXED ? __ldg(js + q2 * p.P1 + p2) :", "")  # kernels during which nobody writes them
    assert not re.findall(r"__ldg\(\s*" + arrays, text)
    assert not re.findall(r"const (?:int|float) \*\s*__restrict__ " + arrays, text)
