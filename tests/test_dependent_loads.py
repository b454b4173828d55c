"""Kernels launched as programmatic dependents are resident while the kernels
before them still write their operands, so they may not read through the
non-coherent path: ld.global.nc (__ldg, or what the compiler makes of
`const T* __restrict__`) is for data that nothing writes in the kernel's
lifetime, and may be moved above griddepcontrol.wait."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_04406_gb300", "csrc")


def _code(path):
    text = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_no_non_coherent_loads():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert files
    found = [(os.path.basename(f), m.group(0)) for f in files
             for m in re.finditer(r"\b__ldg\w*|\bld\.global(?:\.\w+)*\.nc\b|__restrict__?", _code(f))]
    assert not found
