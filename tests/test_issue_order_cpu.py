"""The pair GEMM's two MMA issuers hand the accumulator to each other through a baton barrier.  MMAs of two threads are ordered by
that barrier only between tcgen05 fences, one on either side, and no run shows a missing one: the source is checked."""
import os
import re

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_20586_b200", "csrc", "gemm_pair.cu")


def _unconditional(text):
    """The text without comments and without anything inside braces that open in it."""
    text = re.sub(r"//[^\n]*", "", text)
    out, depth = [], 0
    for c in text:
        depth += (c == "{") - (c == "}")
        if depth == 0:
            out.append(c)
    return "".join(out)


def test_every_step_fences_both_sides_of_the_baton():
    src = open(SOURCE).read()
    take = src.index("mbar_wait_spin(&turn[me]")
    issue = src.index("if (elect_one()) {", take)              # the lane that issues the step's MMAs
    give = src.index("mbar_arrive(&turn[me ^ 1])", issue)
    assert "tc_mma_" in src[issue:give]
    taken = _unconditional(src[src.index("\n", take):issue])
    assert "tc_fence_after_sync();" in taken                   # whatever the step, before its first MMA
    assert "tc_fence_before_sync();" in src[src.rindex("tc_mma_", issue, give):give]      # after its last MMA, before the baton goes on
    assert src.count("mbar_wait_spin(&turn[") == 1 and src.count("mbar_arrive(&turn[") == 1
