"""Packed cell indices (csrc/pack.h) over the range of mesh sides that the
batches accept (n^2 < 2^31), compiled for the host."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "pack.h"
int main() {
    int bad = 0;
    const int c[] = {0, 1, 255, 32767, 32768, 39999, 46338, 46339};
    for (int x : c)
        for (int y : c) {
            const unsigned w = pack_cell(x, y);
            if (cell_x(w) != x || cell_y(w) != y) ++bad;
        }
    for (int x = -30; x <= 30; ++x)
        for (int y = -30; y <= 30; ++y) {
            const unsigned w = pack_offset(x, y);
            if (offset_x(w) != x || offset_y(w) != y) ++bad;
        }
    printf("%d\n", bad);
    return bad != 0;
}
"""


def test_packed_cells_of_the_largest_meshes(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "pack.cpp", tmp_path / "pack"
    src.write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1610_05258_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
