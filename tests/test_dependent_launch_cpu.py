"""Kernels that wait inside for the kernel before them (programmatic dependent launch) read what that kernel may still be writing when
they start.  Nothing but the order of the instructions keeps their loads behind the wait, and no run shows a load that the
compiler was free to move: the source is checked."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_20586_b200", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


WAITING = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and "pdl_wait();" in _code(f))


def test_the_waiting_kernels_are_found():
    assert {"quantize.cu", "quantize_tc.cu", "gemm_pair.cu", "gemm_f8.cu", "variants.cu"} <= set(WAITING)
    assert re.search(r'pdl_wait\(\)\s*{\s*asm volatile\("griddepcontrol\.wait;" ::: "memory"\);', _code("ptx.cuh"))


@pytest.mark.parametrize("name", WAITING)
def test_loads_stay_behind_the_wait(name):
    code = _code(name)
    # loads of data that is promised to be constant while the kernel lives
    assert "__ldg(" not in code and "ld.global.nc" not in code
    # assembly that reads memory, without saying so to the compiler
    for asm in re.findall(r"asm\b[^;{]*\(\s*(?:\"[^\"]*\"\s*)+[^;]*;", code):
        if "ld.global" in asm:
            assert asm.startswith("asm volatile") and '"memory"' in asm, asm
    # pointers that are promised to be the only way to what they point at
    for kernel in code.split("__global__")[1:]:
        if "pdl_wait();" in kernel:
            assert "__restrict__" not in kernel, kernel[:120]
