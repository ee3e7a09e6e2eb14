"""Rules of the kernels' sources that no run would show broken."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_20488_b200", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_nothing_is_read_through_the_read_only_path(path):
    """Kernels are launched while the kernel that writes their inputs still runs.  The read-only path (__ldg, ld.global.nc, and the
    loads a compiler may turn into it behind __restrict__) is for data that does not change while the kernel lives."""
    code = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    assert not re.findall(r"__ldg\b|ld\.global\.nc|__restrict__", code)
