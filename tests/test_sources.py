"""Rules on the kernels' source that no run shows."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1206_5878_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))),
                         ids=os.path.basename)
def test_kernels_under_programmatic_launch_load_coherently(path):
    """A kernel launched programmatically dependent is alive while its predecessor
    writes: the non-coherent load path (memory read-only for the kernel's whole
    life) is not for it."""
    with open(path) as f:
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
    assert not re.findall(r"__ldg|__restrict__|ld\.global\.nc", code)
