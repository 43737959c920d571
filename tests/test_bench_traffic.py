"""The committed DRAM traffic figure is tied to every source that the kernel it
was measured on is compiled from."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1912_03278_gb300", "csrc")


def _included(name, seen):
    for inc in re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, name)).read()):
        if os.path.exists(os.path.join(CSRC, os.path.basename(inc))) and inc not in seen:
            seen.add(inc)
            _included(inc, seen)
    return seen


def test_traffic_sources_are_all_that_the_kernel_includes():
    assert set(bench.TRAFFIC_SOURCES) == {"march_lattice.cu"} | _included("march_lattice.cu", set())
