"""Bounded waits of the tensor-core kernels, by reading their source: no GPU has to run out of time for it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_11498_b200", "csrc")
VOTE = r"__all_sync\(0xffffffffu, ok\)"


def source(kernel):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, kernel + "_sm100.cu")).read())


def enclosing_heads(text, pos):
    """What stands in front of the brace of every block around `pos`, back to the statement before it."""
    heads, last = [], 0
    for m in re.finditer(r"[{};]", text[:pos]):
        if m.group() == "{":
            heads.append(text[last:m.start()])
        elif m.group() == "}":
            heads.pop()
        last = m.end()
    return heads


@pytest.mark.parametrize("kernel", ["attn_fwd", "attn_bwd_dkv", "attn_bwd_dq"])
def test_lanes_of_a_warp_give_up_together(kernel):
    """A lane decides by its own clock that a wait has run out.  In a branch of a whole warp the lanes that go on would wait for the
    ones that left (__syncwarp, tensor-memory accesses) while those wait at the barrier of the block: mbar_wait is for one
    thread, and what mbar_wait_lanes returned is voted on before anything depends on it."""
    text = source(kernel)
    calls = list(re.finditer(r"\bmbar_wait\s*\(", text))
    assert calls   # the producer's
    for m in calls:
        assert any("lane == 0" in h for h in enclosing_heads(text, m.start())), text[m.start():m.start() + 60]
    wait = r"(?:bool )?ok &?= mbar_wait_lanes\("
    assert len(re.findall(wait, text)) == len(re.findall(r"\bmbar_wait_lanes\(", text))
    for m in re.finditer(wait, text):
        use = re.search(r"\bok\b", text[m.end():]).start() + m.end()
        line = text[text.rfind("\n", 0, use) + 1:text.find("\n", use)]
        assert re.search(wait, line) or re.search(r"(ok = |!)" + VOTE, line), line
