"""What the bench states about the sources: the hash that ties the traffic record
to the kernels covers every file that their translation units include, and the
bytes read back for a formula are those that the library copies."""
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


def test_formula_read_is_counted_as_it_is_made():
    """The end-to-end line's device-to-host bytes are those that the library
    copies for a formula of ordinary length."""
    with open(os.path.join(CSRC, "lsyn_api.cu")) as f:
        got = int(re.search(r"size_t got = (\d+);", f.read()).group(1))
    assert bench.FORMULA_READ_BYTES == got + 4


def test_traffic_record_covers_the_kernels_sources():
    need = set()
    for unit in glob.glob(os.path.join(CSRC, "kernels_*.cu")):
        _included(os.path.basename(unit), need)
    assert need and need <= set(bench._kernel_sources())
