"""Kernels start while the kernel before them on the stream still runs
(programmatic dependent launch), so whatever that kernel may have written is
read with coherent loads: no __ldg, no ld.global.nc, and no const __restrict__
parameter of a kernel, which the compiler may turn into one.  The tables of a
grouped plan, which the host fills before any launch, are the exception."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_16080_gb300", "csrc")
PLAN_TABLES = ("unit_group", "tile_start")


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


@pytest.mark.parametrize("name", _sources())
def test_loads_are_coherent(name):
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for m in re.finditer(r"__ldg\(([^\n]*)", code):
        assert any(t in m.group(1) for t in PLAN_TABLES), m.group(0)
    assert "ld.global.nc" not in code
    assert not re.search(r"\bconst\s+[\w:<>]+\s*\*\s*__restrict__", code)
