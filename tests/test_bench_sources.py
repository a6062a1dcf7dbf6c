"""The traffic figures that bench.py reads from a committed profile count only
while the sources of the extraction's kernels are the ones profiled: the hash
covers every file those kernels are built from, and the tables they read."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2009_03254_gb300", "csrc")


def test_profile_hash_covers_the_extractions_sources():
    seen, todo = set(), ["extract.cu", "mc.cu", "mc_tables.cu"]
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        text = open(os.path.join(CSRC, f)).read()
        todo += [i for i in re.findall(r'#include "([^"]+)"', text) if os.path.exists(os.path.join(CSRC, i))]
    assert seen == set(bench.PROFILE_SOURCES)
