"""The tensor-core Gram kernel's promise that a wait that runs out ends the
kernel: its warps leave the panel loop one by one then, so nothing in the loop,
nor in what it calls, may stand in a barrier without a bound (a named barrier
with a thread count would wait for warps that are gone)."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1806_01036_gb300", "csrc",
                   "umma_gram.cu")


def test_panel_loop_has_bounded_waits_only():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    loop = text[text.index("for (; p < npan; ++p) {"):]
    depth = 0
    for i, c in enumerate(loop):
        depth += (c == "{") - (c == "}")
        if c == "}" and depth == 0:
            loop = loop[:i]
            break
    steps = text[text.index("auto issue = ["):text.index("if (npan > 0) {", text.index("auto issue = ["))]
    for part in (loop, steps):
        assert len(part) > 500
        for word in ("__syncthreads", "bar.sync", "bar.red", "barrier"):
            assert word not in part, word
    assert "__all_sync" in loop  # whole warps leave
