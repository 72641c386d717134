"""PTX instructions in their .aligned form have to be reached by all lanes of a
warp together.  In csrc/ each stands in a wrapper of its own; every wrapper puts
a warp barrier in front of it, whatever its callers did before."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2510_02156_gb300", "csrc")
ALIGNED = re.compile(r'asm volatile\(\s*"[^"]*(?:\.aligned\b|\bbar\.sync\b)')


def _functions(text):
    """(name, body) of every function whose definition starts a line."""
    for m in re.finditer(r"^(?:template <[^>]*>\s*)?(?:__device__|__global__)[^;{]*?(\w+)\([^;{]*\)\s*\{", text, re.M):
        depth, i = 1, m.end()
        while depth and i < len(text):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_a_warp_barrier_stands_before_every_aligned_instruction(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    found = 0
    for name, body in _functions(text):
        first = ALIGNED.search(body)
        if first:
            found += len(ALIGNED.findall(body))
            assert "__syncwarp();" in body[:first.start()], name
    assert found == len(ALIGNED.findall(text))
