"""ordered_sum.h at the ends of the float64 range, compiled with checks for undefined
behaviour: the same bits as the loop, and nothing that the language leaves open."""

import os
import shutil
import subprocess

import pytest

SRC = r"""
#include <float.h>
#include <stdio.h>
#include <string.h>
#include "ordered_sum.h"
int main() {
    const double ms[] = {1e303, 3e303, 1.7e304, DBL_MAX / 3, DBL_MAX / 70000, DBL_MAX, 0x1p1000,
                         0x1.8p1010, DBL_MIN, 5e-324, 3e-320};
    const long long ns[] = {1, 2, 3, 70, 1000, 70001, 300000};
    for (double m : ms)
        for (long long n : ns) {
            volatile double a = 0.0;
            for (long long i = 0; i < n; ++i) a = a + m;
            const double x = a, y = sipf::ordered_sum_of_equal(m, n);
            if (memcmp(&x, &y, 8)) {
                printf("%a %lld: %a %a\n", m, n, x, y);
                return 1;
            }
        }
    return 0;
}
"""


def test_sums_near_the_ends_of_the_range(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       "paper_2605_20140_gb300", "csrc")
    exe = tmp_path / "t"
    flags = ["-fsanitize=undefined,float-cast-overflow", "-fno-sanitize-recover=all"]
    build = [cxx, "-O1", "-std=c++17", "-I", inc, str(src), "-o", str(exe)]
    if subprocess.run(build + flags, capture_output=True).returncode:     # no sanitizer here
        subprocess.check_call(build)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
