"""plan_shape.h (host code, compiled here): without room for a cluster the plan kernel
is one block, whatever the grid."""

import os
import shutil
import subprocess

import pytest

SRC = r"""
#include <assert.h>
#include <initializer_list>
#include "plan_shape.h"
int main() {
    for (int T : {1, 2, 3, 4, 6, 8, 9, 12, 16, 18, 24, 27, 32, 36, 48, 54, 64}) {
        const int tiles = T * T * T;
        assert(sipf::plan_blocks(tiles, 0) == 1);
        assert(sipf::plan_blocks(tiles, -1) == 1);
        assert(sipf::plan_blocks(tiles, 1) == (tiles > 1024 ? sipf::kPlanCluster : 1));
        assert(sipf::plan_blocks(tiles, 19) == sipf::plan_blocks(tiles, 1));
    }
    return 0;
}
"""


def test_plan_without_clusters(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       "paper_2605_20140_gb300", "csrc")
    exe = tmp_path / "t"
    subprocess.check_call([cxx, "-O1", "-std=c++17", "-I", inc, str(src), "-o", str(exe)])
    subprocess.check_call([str(exe)])
