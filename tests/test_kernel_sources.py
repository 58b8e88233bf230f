"""What the kernels rely on and no run on a GPU shows: read from their sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_08804_b200", "csrc")


@pytest.mark.parametrize("name", sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu"))))
def test_dynamic_shared_memory_is_aligned(name):
    """Tiles in dynamic shared memory are read and copied 16 bytes at a time (cp.async faults on less), and the static shared variables
    before it end anywhere: it has to be declared so, or its start rounded up by hand."""
    lines = open(os.path.join(CSRC, name)).read().split("\n")
    for i, line in enumerate(lines):
        m = re.search(r"extern __shared__ (?:__align__\((\d+)\) )?[\w ]+ (\w+)\[\];", line)
        assert ("extern __shared__" in line) == bool(m), line
        if m and int(m.group(1) or 0) < 16:
            assert re.search(r"\(uintptr_t\)%s \+ 1023\) & ~\(uintptr_t\)1023" % m.group(2), lines[i + 1]), (name, i + 1, line)
