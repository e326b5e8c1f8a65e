"""Sizes of the scratch that path 1 keeps per stream (host only, no GPU).

A modification by more than 64 vectors runs as launches of 64 and one of what
is left, all in one workspace, and later calls of the same or a smaller size
find the workspace large enough: so the size may fall with neither the order
nor the vector count, and has to hold every launch's layout."""
from __future__ import annotations

import os
import subprocess

import pytest

from paper_1011_1173_gb300 import build as chm_build
from paper_1011_1173_gb300 import chm


@pytest.fixture()
def path1():
    chm.config_set("path", chm.PATH_WAVE)
    yield
    chm.config_set("path", chm.PATH_AUTO)


@pytest.mark.parametrize("dtype", [chm.CHM_F64, chm.CHM_F32_MIXED])
def test_workspace_never_shrinks_with_the_size(path1, dtype):
    for n in (64, 2048, 2049, 4097, 6144, 6145, 7000, 8192, 8193, 12288, 16384, 20000):
        sizes = [chm.workspace_bytes(n, k, dtype) for k in range(1, 70)]
        assert sizes == sorted(sizes), n
    orders = sorted(list(range(1, 17000, 97)) + [2048, 2049, 6144, 6145, 8192, 8193, 12288, 12289, 16384, 16385])
    for k in (1, 2, 3, 8, 9, 16, 17, 58, 64):
        sizes = [chm.workspace_bytes(n, k, dtype) for n in orders]
        assert sizes == sorted(sizes), k


# every (blocks, vectors): the bound holds the layout and never falls
CHECK = r"""
#include "chm_team_layout.h"
using namespace chm;
using namespace chm::team;
int main()
{
    for (int nb = 1; nb <= 600; ++nb)
        for (int k = 1; k <= kMaxWaves; ++k) {
            if (prob_data(nb, k) > prob_data_cap(nb, k)) return 1;
            if (nb > 1 && prob_data_cap(nb - 1, k) > prob_data_cap(nb, k)) return 2;
            if (k > 1 && prob_data_cap(nb, k - 1) > prob_data_cap(nb, k)) return 3;
            if (nb > 1 && (prob_flags(nb - 1, k) > prob_flags(nb, k) || prob_tags(nb - 1, k) > prob_tags(nb, k))) return 4;
            if (k > 1 && (prob_flags(nb, k - 1) > prob_flags(nb, k) || prob_tags(nb, k - 1) > prob_tags(nb, k))) return 5;
        }
    for (int nb = 1; nb <= 4096; ++nb)
        for (int KB = 1; KB <= kTeamKb; KB *= 2) {
            const int b = bounds_of(nb, KB, true);
            if (b < 0 || (size_t)b > bounds_cap(nb, KB) || bounds_of(nb, KB, false) > b) return 6;
        }
    return 0;
}
"""


def test_bound_holds_every_layout(tmp_path):
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", chm_build.SRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
    os.remove(exe)
