"""What one lane of a warp writes to shared memory another may read only after `__syncwarp()` (or a barrier): votes and shuffles
bring the lanes together but order no memory.  The hardware does not show a missing one, so the kernels' text is looked at."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).parent.parent / "paper_2510_07535_b200" / "csrc"


@pytest.mark.parametrize("file,write,read", [
    # the walk: every lane writes its nodes' parents, then follows other lanes'
    ("accept.cuh", r"s_parent\[node\] = parent\[h\];", r"c = s_parent\[c\]"),
])
def test_a_warp_barrier_stands_between_write_and_read(file, write, read):
    text = re.sub(r"//[^\n]*", "", (CSRC / file).read_text())
    between = re.search(write + r"(.*?)" + read, text, re.S).group(1)
    assert "__syncwarp();" in between
