"""A warp copies its job's scene header into shared memory with all lanes,
each some of the words, so nothing may read the copy before the warp has
synchronised: a lane that saw another lane's words too early could leave the
warp's collective operations alone.  No run shows that reliably (the compiler
usually reconverges the warp by itself), so the sources are read."""
import os
import re

import pytest

import paper_2112_08035_gb300 as smc

CSRC = os.path.join(os.path.dirname(smc.__file__), "csrc")
COPY = re.compile(r"reinterpret_cast<long long \*>\(&(\S+?)\);\s*\n\s*for \(int i = lane; .*\) d8\[i\] = s8\[i\];\n")


def _copies(unit):
    with open(os.path.join(CSRC, unit)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    return [(m.group(1), text[m.end():]) for m in COPY.finditer(text)]


@pytest.mark.parametrize("unit,copies", [("smcrt_k64.cu", 1), ("smcrt_k32.cu", 2)])
def test_staged_scene_is_read_after_a_warp_sync(unit, copies):
    found = _copies(unit)
    assert len(found) == copies
    for name, rest in found:
        sync = rest.find("__syncwarp()")
        read = re.search(re.escape(name) + r"\b", rest)
        assert sync >= 0 and (read is None or sync < read.start()), (unit, name)
