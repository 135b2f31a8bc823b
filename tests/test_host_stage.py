"""host_stage.h (host code, compiled here): where memory cannot be pinned the
staging buffer is ordinary memory, and each kind is given back as it was taken."""

import os
import shutil
import subprocess

import pytest

SRC = r"""
#include <assert.h>
#include <string.h>
#include "host_stage.h"
int main() {
    int pins = 0, unpins = 0;
    auto pin = [&](void** q, size_t bytes) { ++pins; *q = malloc(bytes); return true; };
    auto refuse = [&](void** q, size_t) { ++pins; *q = nullptr; return false; };
    auto unpin = [&](void* q) { ++unpins; free(q); };
    // pinned at once, on the second call, never; where that can be had and where not
    for (int when = 0; when < 3; ++when)
        for (int can = 0; can < 2; ++can) {
            sipf::HostStage s;
            pins = unpins = 0;
            for (int call = 0; call < 3; ++call) {
                assert(can ? s.get(1000, when == 0, when == 1, pin)
                           : s.get(1000, when == 0, when == 1, refuse));
                assert(s.p && s.pinned == (can && when <= call && when < 2));
                memset(s.p, 1, 1000 * sizeof(double));
            }
            assert(pins == (when < 2));
            s.release(unpin);
            assert(!s.p && unpins == (can && when < 2));
            s.release(unpin);                     // nothing left
            assert(unpins == (can && when < 2));
        }
    sipf::HostStage none;
    assert(!none.get(size_t{1} << 60, true, true, refuse) && !none.p);
    return 0;
}
"""


def test_staging_buffer_without_pinned_memory(tmp_path):
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
