"""Kernels that may start as programmatic dependents read global memory with ordinary loads.

Such a kernel is resident while the kernel before it in the stream still writes, so what that kernel wrote is not
read-only for its lifetime, which the read-only path (__ldg, ld.global.nc) asks for; the compiler may also move
such a load ahead of griddepcontrol.wait.  A stale value would be rare and would depend on timing, so that the sources
are checked instead."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2006_16236_b200", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


@pytest.mark.parametrize("name", ["la_mma.cuh", "la_mma_sweep.cuh", "la_causal_mma.cu", "la_linear_mma.cu"])
def test_no_read_only_loads(name):
    assert not re.findall(r"__ldg\s*\(|ld\.global\.nc|__restrict__", _code(name))
