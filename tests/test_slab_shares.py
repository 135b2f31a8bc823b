"""slab_shares.h (host code, compiled here): with any number of SMs the allocation-free
deposit launches a block for every slab, so that the kernel's rule -- one each, the
rest in proportion to a slab's work -- leaves none out."""

import os
import shutil
import subprocess

import pytest

SRC = r"""
#include <assert.h>
#include <stdint.h>
#include <stdlib.h>
#include <vector>
#include "slab_shares.h"
using namespace sipf;
struct Share { int slab, part, parts; };
// k_na_slab's rule for one block
static Share slab_share(int block, int grid, int H, int64_t N, const unsigned long long* planes) {
    const int P = slab_planes(H), slabs = slab_count(H);
    double all = 0.0;
    for (int k = 0; k < H; ++k) all += double(planes[k]);
    const double scan = N / 24.0, total = all + scan * slabs;
    Share s{-1, 0, 0};
    int first = 0;
    for (int b = 0; b < slabs; ++b) {
        double n = scan;
        for (int k = b * P; k < (H < (b + 1) * P ? H : (b + 1) * P); ++k) n += double(planes[k]);
        const int r = 1 + int((grid - slabs) * (n / total));
        const int id = block - first;
        if (id >= 0 && id < r) s = Share{b, id, r};
        first += r;
    }
    return s;
}
int main() {
    srand(1);
    for (int H = 1; H <= 64; ++H) {
        const int P = slab_planes(H), slabs = slab_count(H);
        assert(P >= 1 && (slabs - 1) * P < H && slabs * P >= H);
        assert((P + 1) * H * H * 8 <= kSlabBytes || P == H);
        for (int sms : {1, 2, 7, 12, 13, 14, 76, 148, 152}) {
            const int grid = slab_grid(sms, H);
            assert(grid >= sms && grid >= slabs);
            for (int shape = 0; shape < 4; ++shape) {
                // even, one plane holds all, none counts (bad masses), random
                std::vector<unsigned long long> planes(H, 0);
                const int64_t N = 1 << 20;
                for (int k = 0; k < H; ++k)
                    planes[k] = shape == 0 ? N / H : shape == 1 ? (k == H / 2 ? N : 0)
                              : shape == 2 ? 0 : rand() % (N / H + 1);
                std::vector<std::vector<int>> seen(slabs);
                for (int b = 0; b < grid; ++b) {
                    const Share s = slab_share(b, grid, H, N, planes.data());
                    if (s.slab < 0) continue;
                    assert(s.slab < slabs && s.part >= 0 && s.part < s.parts);
                    seen[s.slab].resize(s.parts);
                    assert(seen[s.slab][s.part]++ == 0);
                }
                for (auto& v : seen) {
                    assert(!v.empty());
                    for (int n : v) assert(n == 1);
                }
            }
        }
    }
    return 0;
}
"""


def test_every_slab_has_its_blocks(tmp_path):
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
