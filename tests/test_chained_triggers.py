"""The step's kernels are launched programmatically, but none of them lets the
next one in before it exits: the next one's CTAs would take whatever room is
left, many of them on one SM, and wait there, and their work be spread unevenly
(FP64 steps took up to 2.6 times as long).  Checked in the source; the colour
passes of a sweep (mg.cu) do, whose CTAs have work of their own before the wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2008_11520_gb300", "csrc")


@pytest.mark.parametrize("file", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")) and f != "mg.cu"))
def test_no_early_trigger(file):
    with open(os.path.join(CSRC, file)) as f:
        src = re.sub(r"//.*", "", f.read())
    helper = r"__device__ __forceinline__ void pdl_trigger\(\).*"   # its definition
    src = re.sub(helper, "", src)
    assert not re.search(r"\bpdl_trigger\(|griddepcontrol\.launch_dependents", src), file
