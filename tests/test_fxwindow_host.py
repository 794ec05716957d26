"""The pull gathers' windowed sums equal the sums of the shares' 128-bit
conversions, over every span a window takes, with zeros of both signs and
as many terms as a work item has."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fxwin") / "libfxwin.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off",
                    "-Wno-attributes", os.path.join(HERE, "fxwindow_host.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def test_windows_by_span(lib):
    # a degree bound of 2^18 leaves 127 - 18 - 53 = 56 bits of span exact
    assert [lib.win_windows(900, 900 + s, 18) for s in (0, 31, 32, 55, 56, 57, 63, 64, 200)] == [
        1, 1, 2, 2, 2, 0, 0, 0, 0]
    assert lib.win_windows(0, 5, 18) == 0          # a subnormal share
    assert lib.win_windows(2047, 0, 18) == 0       # no shares
    assert lib.win_windows(1985, 1990, 18) == 0


@pytest.mark.parametrize("n", [1, 7, 256, 4096])
@pytest.mark.parametrize("be_min", [1, 37, 993, 1984])
@pytest.mark.parametrize("span", [0, 1, 31, 32, 33, 56])
def test_sums(lib, n, be_min, span):
    rng = np.random.default_rng(span * 7 + be_min + n)
    w = lib.win_windows(be_min, be_min + span, 12)
    assert w == (1 if span < 32 else 2)
    for fill in ("random", "ones"):
        m = (rng.integers(0, 1 << 52, n, dtype=np.int64) if fill == "random"
             else np.full(n, (1 << 52) - 1, np.int64))
        be = rng.integers(be_min, be_min + span + 1, n)
        if fill == "ones":
            be[:] = be_min + span  # the largest sums
        x = ((be.astype(np.int64) << 52) | m).view(np.float64)
        x[rng.random(n) < 0.2] = 0.0
        x[rng.random(n) < 0.05] = -0.0
        assert lib.win_differs(w, ctypes.c_int64(n), ctypes.c_void_p(x.ctypes.data), be_min,
                               be_min + span, 12) == 0
