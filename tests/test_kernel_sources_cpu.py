"""Properties of the kernel sources that no run shows while the compiler happens to place
things well."""
from __future__ import annotations

import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_dynamic_shared_memory_is_declared_for_16_byte_accesses():
    """Parts of the dynamic shared arrays are read and written as 16-byte vectors, and static
    shared variables may lie in front of them: the declaration asks for the alignment."""
    found = 0
    for path in glob.glob(os.path.join(ROOT, "paper_2009_07914_gb300", "csrc", "*.cu*")):
        for line in open(path):
            if re.match(r"\s*extern\s+__shared__", line):
                found += 1
                assert "__align__(16)" in line, (path, line)
    assert found >= 5
