"""What one lane of a warp writes to shared memory another may read, and what it reads another may overwrite, only after
`__syncwarp()` (or a barrier): votes and shuffles bring the lanes together but order no memory.  The hardware does not show a
missing one, so the kernels' text is looked at."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).parent.parent / "paper_2510_07535_b200" / "csrc"


@pytest.mark.parametrize("file,first,then", [
    # the walk: every lane writes its nodes' parents, then follows other lanes'
    ("accept.cuh", r"s_parent\[node\] = parent\[h\];", r"c = s_parent\[c\]"),
    # the merge: each round of each block puts LSEs where other lanes have read the weights of the one before
    ("combine.cuh", r"for \(int base = 0; base < count; base \+= group\) \{", r"cp\.async\.cg"),
])
def test_a_warp_barrier_stands_between(file, first, then):
    text = re.sub(r"//[^\n]*", "", (CSRC / file).read_text())
    between = re.search(first + r"(.*?)" + then, text, re.S).group(1)
    assert re.search(r"\n\s*__syncwarp\(\);", between)          # unconditional: a line of its own
