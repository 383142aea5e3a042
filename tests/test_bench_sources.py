"""bench.py's list of the sources behind each timed kernel (its committed counters count only while those are
unchanged), on CPU: the list names every header that the kernel's translation unit includes, directly or through
another, apart from the one that only declares host functions, the API header and the generated tables (the
generator stands for them)."""
import os
import re
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))

import bench  # noqa: E402

CSRC = os.path.join(os.path.dirname(HERE), "paper_2312_02756_gb300", "csrc")


def _included(name, seen):
    with open(os.path.join(CSRC, name)) as f:
        for inc in re.findall(r'^#include "([^"]+)"', f.read(), re.M):
            if inc not in seen and os.path.exists(os.path.join(CSRC, inc)):
                seen.add(inc)
                _included(inc, seen)
    return seen


@pytest.mark.parametrize("kernel", sorted(bench.KERNEL_SOURCES))
def test_every_header_is_listed(kernel):
    listed = bench.KERNEL_SOURCES[kernel]
    unit = listed[0]
    assert unit.endswith(".cu")
    assert _included(unit, {unit}) - {"gvx_internal.h"} <= set(listed)
