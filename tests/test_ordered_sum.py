"""ordered_sum.h against plain loops (host code, compiled here): the sum of n
equal masses has the bits of n additions in a row, and any_order_exact only
says yes where every order of addition gives one value."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

SRC = r"""
#include "ordered_sum.h"
extern "C" double of_equal(double m, long long n) { return sipf::ordered_sum_of_equal(m, n); }
extern "C" double one_by_one(double m, long long n) {
    double a = 0.0;
    for (long long i = 0; i < n; ++i) a += m;
    return a;
}
extern "C" int any_order(long long n, double m, int low) { return sipf::any_order_exact(n, m, low); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("ordered_sum")
    src = d / "t.cpp"
    src.write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                       "paper_2605_20140_gb300", "csrc")
    out = d / "t.so"
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", inc, str(src), "-o",
                           str(out)])
    lib = ctypes.CDLL(str(out))
    for f in (lib.of_equal, lib.one_by_one):
        f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double, ctypes.c_longlong]
    lib.any_order.argtypes = [ctypes.c_longlong, ctypes.c_double, ctypes.c_int]
    return lib


def test_sum_of_equal_values_has_the_bits_of_the_loop(lib):
    rng = np.random.default_rng(5)
    cases = [(1.0 / n, n) for n in (1, 2, 3, 1000, 65535, 65536, 200003, 1 << 22)]
    # halfway cases (short mantissas), denormals, overflow
    cases += [((2.0 ** b + 1) * 2.0 ** -40, n) for b in range(1, 40, 3) for n in (7, 1000, 65537)]
    cases += [((2.0 ** 52 + 1) * 2.0 ** -90, 300001), (5e-324, 100000), (1e-310, 100003),
              (1.7e308, 5)]
    cases += [(float(np.ldexp(rng.uniform(0.5, 1.0), int(rng.integers(-60, 20)))),
               int(np.exp(rng.uniform(0.0, np.log(3e5))))) for _ in range(400)]
    for m, n in cases:
        assert lib.of_equal(m, n) == lib.one_by_one(m, n), (m, n)


def test_any_order_exact_is_exact(lib):
    rng = np.random.default_rng(6)
    for low in (-30, -25, -3):
        x = (rng.integers(1, 1 << 20, 4096) * 2.0 ** low).astype(np.float64)
        assert lib.any_order(x.size, float(x.max()), low)
        assert len({float(np.cumsum(rng.permutation(x))[-1]) for _ in range(4)}) == 1
    assert not lib.any_order(1 << 22, 1.0, -32)      # partial sums of up to 54 bits
    assert lib.any_order(1 << 22, 1.0, -31)
