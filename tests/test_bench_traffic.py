"""The benchmark reports a recorded DRAM traffic of the plane kernel only while
its sources are unchanged: they are every file the kernel is compiled from and
the one that plans its launch."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1406_4960_gb300", "csrc")


def _included(name, seen):
    if name not in seen and os.path.isfile(os.path.join(CSRC, name)):
        seen.add(name)
        for inc in re.findall(r'#include "([^"/]+)"', open(os.path.join(CSRC, name)).read()):
            _included(inc, seen)
    return seen


def test_plane_sources_cover_kernel_and_plan():
    assert _included("rowspace32.cu", set()) | {"apply.cu"} <= set(bench.PLANE_SOURCES)
