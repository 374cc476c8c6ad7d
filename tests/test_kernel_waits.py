"""Bounded waits of the kernels, by their sources (no GPU): a wait can expire for some lanes of a warp
before others, so every wait outside the regions of one thread either decides nothing or is decided for
the warp as a whole, before warp-wide instructions that need all lanes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1507_08157_gb300", "csrc")
ONE_THREAD = re.compile(r"elect_one\(\)|lane == 0|threadIdx\.x == 0|__device__ __forceinline__ bool mma_block")


def _enclosing(text, at):
    """Headers of the blocks around a position: the text between a block's brace and the statement before."""
    depth, out, i = 0, [], at
    while i > 0:
        i -= 1
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth:
                depth -= 1
            else:
                out.append(text[max(text.rfind(c, 0, i) for c in ";{}") + 1:i])
    return out


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith(".cu")))
def test_waits_of_whole_warps_are_votes(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    for m in re.finditer(r"\bmbar_wait\(", text):
        statement = text[max(text.rfind(c, 0, m.start()) for c in ";{}") + 1:m.start()]
        alone = any(ONE_THREAD.search(h) for h in _enclosing(text, m.start()))
        # a wait whose result decides nothing (the warp walks on, without waiting once the kernel gave up)
        dropped = re.fullmatch(r"\s*(if \([^!]*\)\s*)?", statement) and re.match(r"mbar_wait\([^;]*wlim\);", text[m.start():])
        assert alone or dropped or "__all_sync(0xffffffffu, " in statement, text[m.start() - 80:m.start() + 60]
