"""Rules that every kernel source keeps and no run of a kernel shows reliably."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_23608_b200", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def code(name):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)


@pytest.mark.parametrize("name", FILES)
def test_no_load_can_move_above_the_wait_for_the_kernel_before(name):
    """Kernels start while those before them still run (programmatic dependent launch): a load that the compiler may take
    for one of constant memory can be served before the writer is done."""
    text = code(name)
    assert not re.search(r"ld\.global(\.\w+)*\.nc", text)
    # but for a linear layer's bias: a parameter, read under a branch on what was read behind the wait
    assert not re.search(r"\b__ld(g|cg|ca|cs|lu|cv)\s*\((?!reinterpret_cast<const uint4\*>\(bias \+ col\)\))", text)
    assert not re.search(r"\bconst\s+[\w:]+\s*\*\s*(const\s+)?__restrict__", text)
    for load in re.findall(r"asm\s+(\w*)\s*\(\s*\"ld\.global", text):
        assert load == "volatile"
    # an array that one pass of a kernel writes and another only reads
    assert not re.search(r"__restrict__\s+delta\b", text)
