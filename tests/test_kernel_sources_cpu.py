"""CPU checks of the CUDA sources: inline instructions that a warp must execute
as a whole (the aligned forms in inline PTX, which the compiler does not treat
as convergence points) follow a __syncwarp() where lanes can have parted."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_09432_gb300", "csrc")


def code_lines(name):
    """The file's lines without comments and blank lines."""
    src = open(os.path.join(CSRC, name)).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    lines = [re.sub(r"//.*", "", ln).strip() for ln in src.splitlines()]
    return [ln for ln in lines if ln]


@pytest.mark.parametrize("name,instruction", [("vec_kernel.cuh", "bar.arrive"), ("lbpf_nn.cu", "tcgen05.ld.sync")])
def test_warp_is_converged_before(name, instruction):
    lines = code_lines(name)
    found = 0
    for k, ln in enumerate(lines):
        if instruction not in ln:
            continue
        found += 1
        k -= lines[k - 1].startswith("asm volatile(")  # the instruction's text on its own line
        assert lines[k - 1] == "__syncwarp();", f"{name}: {ln}"
    assert found > 0
