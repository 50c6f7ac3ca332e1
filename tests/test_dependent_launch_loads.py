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


READ_ONLY = r"__ldg\s*\(|ld\.global\.nc|const \w+\s*\*\s*__restrict__"


NO_READ_ONLY_LOADS = ["la_mma.cuh", "la_mma_sweep.cuh", "la_causal_mma.cu", "la_linear_mma.cu", "la_tc_common.cuh", "la_tc_causal_fwd.cu",
                      "la_tc_causal_bwd.cu", "la_tc_segment.cu", "la_tc_linear.cu", "la_decode_layer.cu", "la_sm100.cuh", "la_cluster.cu", "la_common.cuh", "la_tc.cuh"]


@pytest.mark.parametrize("name", NO_READ_ONLY_LOADS)
def test_no_read_only_loads(name):
    assert not re.findall(READ_ONLY, _code(name))


def test_the_chained_kernel_of_the_elementwise_file():
    code = _code("la_elementwise.cu")
    kernels = {re.search(r"(\w+_kernel)\(", k).group(1): k for k in code.split("__global__")[1:]}
    chained = [n for n, k in kernels.items() if "griddepcontrol.wait" in k]
    assert chained == ["recurrent_step_kernel"]
    assert not re.findall(READ_ONLY, kernels[chained[0]].split("template")[0])


def test_no_other_file_launches_programmatic_dependents():
    known = {"la_mma_sweep.cuh", "la_tc_common.cuh", "la_elementwise.cu"}       # where the launch attribute is set
    assert {n for n in os.listdir(CSRC) if "ProgrammaticStreamSerialization" in _code(n)} == known
    by_helper = {n for n in os.listdir(CSRC) if re.search(r"\bchained_launch\s*\(", _code(n))}
    assert by_helper == {"la_tc_common.cuh", "la_cluster.cu", "la_decode_layer.cu", "la_tc_causal_bwd.cu", "la_tc_causal_fwd.cu", "la_tc_linear.cu",
                         "la_tc_segment.cu"}
    waits = {n for n in os.listdir(CSRC) if re.search(r"\b(grid_dependency_wait|wait_for_stream)\s*\(|griddepcontrol\.wait", _code(n))}
    assert waits - {"la_elementwise.cu"} <= set(NO_READ_ONLY_LOADS)
