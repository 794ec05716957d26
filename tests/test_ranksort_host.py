"""Which sorts count, at the rule's edge and where n * n leaves 64 bits."""
import ctypes
import math
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def takes(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("ranksort") / "libranksort.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared",
                    os.path.join(HERE, "ranksort_host.cpp"), "-o", so], check=True)
    f = ctypes.CDLL(so).rank_takes
    f.argtypes = [ctypes.c_int64, ctypes.c_int]
    return lambda n, d: bool(f(n, d))


@pytest.mark.parametrize("digits", [1, 2, 3, 4, 5, 8])
def test_rule(takes, digits):
    edge = math.isqrt(digits * (50 << 20))
    sizes = [0, 1, 2, 1025, edge - 1, edge, edge + 1, 2 * edge, 1 << 31, (1 << 31) + 1,
             3_037_000_499, 3_037_000_500, 3_100_000_000, 4_294_967_295, 4_294_967_296,
             4_294_967_297, 5_500_000_000, 6_074_001_000, 1 << 33, 1 << 40, 1 << 62]
    for n in sizes:
        assert takes(n, digits) == (n * n <= digits * (50 << 20)), n
