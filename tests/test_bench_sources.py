"""The benchmark's record of DRAM traffic is keyed by the sources of the ASK
kernels: all of them."""
import os
import re

import bench

CSRC = "paper_2206_02255_gb300/csrc"


def _included(name, seen):
    if name not in seen:
        seen.add(name)
        for inc in re.findall(r'^#include "([^"/]+)"', open(os.path.join(bench.ROOT, CSRC, name)).read(), re.M):
            _included(inc, seen)
    return seen


def test_traffic_key_covers_the_kernel_sources():
    want = {"%s/%s" % (CSRC, f) for f in _included("ask_kernels.cu", set())}
    assert want == set(bench.KERNEL_SOURCES)
