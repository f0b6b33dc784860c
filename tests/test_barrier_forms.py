"""Barriers in inline PTX: the forms that need every lane of a warp converged
(`.aligned`, and `bar.*`, which implies it) are undefined after code whose
lanes diverge, and nothing tells the compiler to reconverge them there.  The
kernels reach their barriers from such code (lanes without a neuron, loops of
uneven length), so they use the other forms."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1906_03958_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_inline_barriers_need_no_converged_warp(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    ptx = " ".join(re.findall(r'"((?:[^"\\]|\\.)*)"', text))
    barriers = re.findall(r"\b(?:bar|barrier)\.[\w.:]+", ptx)
    assert not [b for b in barriers if b.startswith("bar.") or ".aligned" in b]
