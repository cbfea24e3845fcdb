"""The hash that ties the sweep's profiles to its source covers every file the
sweep kernels are compiled from."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1204_5072_gb300", "csrc")


def test_hash_covers_the_includes():
    todo, files = ["kpz_sweep.cu"], set()
    while todo:
        f = todo.pop()
        if f not in files:
            files.add(f)
            todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, f)).read())
    assert set(bench.SWEEP_SOURCES) == files
