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


@pytest.mark.parametrize("name,kernel,waiting", [("tc_fwd.cu", "k_tc_chain_fwd", 5), ("tc_fwd.cu", "k_tc_chain_fwd_half", 6),
                                                 ("tc_bwd.cu", "k_tc_chain_bwd", 4), ("tc_bwd.cu", "k_tc_chunk_bwd", 3)])
def test_bounded_waits_begin_after_the_kernel_before(name, kernel, waiting):
    """A CTA may start while the kernel before it runs, for as long as that takes; the time limit of a wait inside the CTA is meant for the
    CTA's own work, so every role of its warps waits for that kernel before its first bounded wait: always, or whatever a flag says, or
    (p.beside, see sm100.cuh) unless the launch depends on nothing of it."""
    src = open(os.path.join(CSRC, name)).read()
    body = src[re.search(r"__global__ [^;{]*\b%s\(" % kernel, src).end():]
    body = body[:body.index("\n}\n")]
    roles = re.split(r"\n *// (?:-{10,}|={10,}) (.+?) (?:-{10,}|={10,})\n", body)
    assert len(roles) >= 9, kernel
    found = 0
    for role, text in zip(roles[1::2], roles[2::2]):
        first = re.search(r"\bwait[()]", text)          # called, or handed on
        if first is None:
            continue
        found += 1
        before = text[:first.start()]
        flags = re.findall(r"^ *if \((!?)p\.(\w+)\) grid_dep_wait\(\);", before, re.M)
        assert re.search(r"^ *grid_dep_wait\(\);", before, re.M) or ("!", "beside") in flags or \
            any(("!", f) in flags and ("", f) in flags for _, f in flags), (kernel, role)
    assert found == waiting, (kernel, found)
