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


@pytest.mark.parametrize("kernel", ["attn_fwd_simt_kernel", "attn_bwd_simt_kernel"])
@pytest.mark.parametrize("has_tile", [True, False])
def test_own_rows_have_landed_before_the_barrier_that_publishes_them(kernel, has_tile):
    """fp32 attention: a thread's own rows are its oldest group of asynchronous copies.  The wait in front of the barrier leaves
    the newest n groups in flight, which must not be all that a thread without a streamed tile (segments of one) has."""
    text = code("attn_simt.cu")
    body = text[text.index(kernel + "("):]
    body = body[:body.index("for (int t = grp; t < n_tiles")]
    staging = re.search(r"auto stage = \[&\]\(int t\) \{(.*?)\n  \};", body, re.S)
    assert body[:staging.start()].count("cp_async_commit();") == 1
    rest = body[staging.end():]
    assert len(re.findall(r"if \(grp < n_tiles\) stage\(grp\);", rest)) == 1 and "cp_async_commit" not in rest
    committed = 1 + (staging.group(1).count("cp_async_commit();") if has_tile else 0)
    helper = re.search(r"void own_rows_landed\(bool has_tile\) \{(.*?)\n\}", text, re.S)
    if helper:
        branch = re.sub(r"\s+", " ", helper.group(1)).strip()
        assert branch == "if (has_tile) cp_async_wait<kBehind>(); else cp_async_wait<0>(); __syncthreads();"
    left = None
    for wait in re.finditer(r"cp_async_wait<(\d)>\(\);|own_rows_landed<(\d)>\(grp < n_tiles\);", rest):
        left = int(wait.group(1)) if wait.group(1) else int(wait.group(2)) if has_tile else 0
    assert left is not None and left < committed


@pytest.mark.parametrize("name", FILES)
def test_a_warp_comes_together_before_one_lane_arrives_for_it(name):
    """An arrival orders what its own thread did.  What the other lanes did (loads of TMEM that the next product overwrites, stores
    that it reads) is ordered by the barrier among them in front of it."""
    for before in re.findall(r"([^;{}]*[;{}])\s*if \(lane == 0\) \{?\s*ptx::mbar_arrive\(", code(name)):
        assert re.fullmatch(r"\s*(__syncwarp\(\)|ptx::named_barrier\([^;]*\));", before), before
