"""Sources of the kernels that may start before the grid in front of them has
ended (launch_next): `__ldg`, and `__restrict__` on data that a kernel only
reads, let the compiler use the read-only load, which asks that the data not
change while the kernel runs, and such a kernel runs while its inputs are still
being written.  (Arrays that the kernel writes itself may be `__restrict__`.)"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_01444_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


FILES = [f for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))) if "launch_next(" in _code(f)]


def test_the_sources_are_found():
    assert FILES


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_no_read_only_loads_where_launches_overlap(path):
    read_only = r"__ldg\b|\bconst\b[^,;(){}]*__restrict__|ld\.global(?:\.\w+)*\.nc\b"
    assert re.findall(read_only, _code(path)) == []
