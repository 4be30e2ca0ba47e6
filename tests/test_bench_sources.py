"""bench.py keys captured traffic and instruction counts by a hash of the step's sources: every
header that the step includes, and the file that picks its tiles, must be among them."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2206_11637_gb300", "csrc")


def included(name, seen):
    if name not in seen:
        seen.add(name)
        with open(os.path.join(CSRC, name)) as f:
            for other in re.findall(r'^#include "([^"]+)"', f.read(), re.M):
                included(other, seen)
    return seen


def test_hashed_sources_cover_the_step():
    need = included("step.cuh", set()) | {"pflbm.cu"}
    assert need <= set(bench.KERNEL_SOURCES), need - set(bench.KERNEL_SOURCES)
