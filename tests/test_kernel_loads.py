"""Sources of the kernels that may start before the grid in front of them has
ended (launch_next): `__ldg` and `__restrict__` let the compiler use the
read-only load, which asks that the data not change while the kernel runs, and
such a kernel runs while its inputs are still being written."""
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
    assert re.findall(r"__ldg\b|__restrict__\b|ld\.global(?:\.\w+)*\.nc\b", _code(path)) == []
