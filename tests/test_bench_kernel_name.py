"""bench.py names the kernel that path 1 runs by its own copy of the library's
size rule (for its output only): the copy has to agree with the source."""
from __future__ import annotations

import os
import re

import bench

SRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_1011_1173_gb300", "csrc", "chm_modify.cu")


def ranges(name):
    text = open(SRC).read()
    body = re.search(r"TeamRange %s\[\] = \{(.*)\};" % name, text).group(1)
    return [(int(n), 64 if k == "kMaxWaves" else int(k)) for n, k in re.findall(r"\{(\d+), (\w+)\}", body)]


def test_bench_names_the_kernel_that_runs():
    for mixed, name in ((False, "kTeamF64"), (True, "kTeamF32")):
        table = ranges(name)
        assert table
        for n in sorted({m + d for m, _ in table for d in (-1, 0, 1)} | {1, 512, 5000, 32768}):
            for k in (1, 2, 4, 5, 8, 9, 16, 17, 64, 100):
                assert bench.team_kernel_takes(n, k, mixed) == any(n <= m and min(k, 64) <= c for m, c in table), (n, k)
