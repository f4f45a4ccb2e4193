"""The compositor's captured DRAM traffic is reported only for the sources it was
taken on: the hash covers the kernel and the library's headers that it includes."""
import os
import re

import bench

CSRC = "paper_2604_25459_gb300/csrc/"


def _included(name, seen):
    seen.add(name)
    with open(os.path.join(bench.ROOT, CSRC, name)) as f:
        for inc in re.findall(r'#include "([^"]+)"', f.read()):
            if inc not in seen and os.path.exists(os.path.join(bench.ROOT, CSRC, inc)):
                _included(inc, seen)
    return seen


def test_traffic_hash_covers_the_compositor():
    assert set(bench.COMPOSITE_TRAFFIC_SOURCES) == {CSRC + f for f in _included("gs_composite.cu", set())}
    assert len(bench._sources_sha(bench.COMPOSITE_TRAFFIC_SOURCES)) == len(bench.COMPOSITE_TRAFFIC_SHA)
