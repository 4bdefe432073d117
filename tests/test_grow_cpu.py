"""A growing device table after an allocation that failed (CPU only: a fake allocator)."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

PROGRAM = r"""
#include <cstdlib>
#include "grow.h"
int main() {
    int *p = nullptr, calls = 0, freed = 0;
    size_t cap = 0;
    bool fails = false;
    auto alloc = [&](int **q, size_t bytes) { ++calls; *q = fails ? nullptr : (int *)malloc(bytes); return !fails; };
    auto release = [&](int *q) { if (q) ++freed; free(q); };
    if (!phia::grow_table(p, cap, 100, alloc, release) || !p || cap != 100) return 1;
    int *first = p;
    if (!phia::grow_table(p, cap, 50, alloc, release) || p != first || calls != 1) return 2;
    fails = true;
    if (phia::grow_table(p, cap, 200, alloc, release) || p || cap || freed != 1) return 3;
    fails = false;
    if (!phia::grow_table(p, cap, 50, alloc, release) || !p || cap != 50 || calls != 3) return 4;
    free(p);
    return 0;
}
"""


def test_a_failed_growth_leaves_no_capacity(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "grow.cpp", tmp_path / "grow"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2407_10205_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)]).returncode == 0
