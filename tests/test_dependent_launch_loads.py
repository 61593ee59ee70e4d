"""Loads of programmatic dependent launches (source check, on the CPU).

Such a kernel starts while the kernel that writes its inputs still runs.  The
non-coherent path (ld.global.nc, which the compiler may also choose for
const __restrict__ parameters and need not keep behind griddepcontrol.wait) asks
for memory that nobody writes during the kernel's whole life, so it is left to
constants: weights of the prompt kernels, norm gains, the rotation table and the
token ids uploaded before the first launch.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_08168_gb300", "csrc")
CONSTANTS = {"embed", "toks", "g"}  # parameters that may be const __restrict__
LDG = ("reinterpret_cast<const uint2*>(g)", "a.rope")  # what __ldg may read


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", ["gemm.cu", "prefill.cu", "tc_gemm.cuh"])
def test_no_non_coherent_loads_of_written_memory(name):
    src = source(name)
    assert "griddepcontrol" in source("ssd_internal.cuh") and "pdl_wait()" in src
    assert "global.nc" not in src
    for m in re.finditer(r"__ldg\(", src):
        assert src[m.end():].startswith(LDG), src[m.start():m.start() + 80]
    params = re.findall(r"const [\w:]+\s*\*\s*__restrict__\s+(\w+)", src)
    assert set(params) <= CONSTANTS, params
