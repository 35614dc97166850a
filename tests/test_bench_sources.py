"""The recorded DRAM traffic that bench.py reports belongs to the kernel sources it was counted
with: every file of this repository that those sources include is part of the key."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2601_03935_gb300", "csrc")


def test_traffic_key_covers_every_included_source():
    seen, todo = set(), [bench.KERNEL_SOURCES[0]]
    while todo:
        name = todo.pop()
        if name in seen:
            continue
        seen.add(name)
        text = open(os.path.join(CSRC, name)).read()
        todo += [x for x in re.findall(r'^#include "([^"/]+)"', text, re.M)]
    assert seen == set(bench.KERNEL_SOURCES)
