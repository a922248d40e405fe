"""The bench's traffic record holds for the sources it was taken from: the hash
that says so covers every file that the kernels' translation units include."""
from __future__ import annotations

import glob
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_2504_18943_gb300", "csrc")


def _included(name, seen):
    with open(os.path.join(CSRC, name)) as f:
        for inc in re.findall(r'#include "([^"]+)"', f.read()):
            if inc not in seen and os.path.exists(os.path.join(CSRC, inc)):
                seen.add(inc)
                _included(inc, seen)
    return seen


def test_traffic_record_covers_the_kernels_sources():
    need = set()
    for unit in glob.glob(os.path.join(CSRC, "kernels_*.cu")):
        _included(os.path.basename(unit), need)
    assert need and need <= set(bench._kernel_sources())
