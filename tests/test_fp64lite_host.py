"""The short forms of fp64lite.cuh equal the expressions they stand for, in
every case: thresholds next to the compared value, small and large degrees,
constants outside the single-precision range, quotients next to a midpoint."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fp64lite") / "libfp64lite.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off",
                    "-Wno-attributes", os.path.join(HERE, "fp64lite_host.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def bad(fn, *arrays):
    fn.restype = ctypes.c_int64
    return fn(ctypes.c_int64(len(arrays[0])), *[ctypes.c_void_p(a.ctypes.data) for a in arrays])


def degrees(rng, n):
    d = np.exp(rng.uniform(0, np.log(2.0 ** 31 - 1), n)).astype(np.int64)
    return np.clip(d, 1, 2 ** 31 - 1).astype(np.int32)


@pytest.mark.parametrize("lo,hi", [(-12, 0), (-40, -20), (15, 25), (-300, 250)])
def test_reaches(lib, lo, hi):
    rng = np.random.default_rng(lo + 500)
    n = 400_000
    c = 10.0 ** rng.uniform(lo, hi, n)
    d = degrees(rng, n)
    t = c * d.astype(np.float64)
    near = t.copy()
    k = rng.integers(-3, 4, n)
    bits = near.view(np.int64) + k * np.where(rng.random(n) < 0.5, 1, 1 << 32)
    near = bits.view(np.float64)  # within a few units of the last place, or of the high word
    far = t * 10.0 ** rng.uniform(-6, 6, n)
    for x in (t, near, far, np.zeros(n), np.full(n, 5e-324)):
        assert bad(lib.reaches_bad, np.ascontiguousarray(x), c, d) == 0


@pytest.mark.parametrize("lo,hi", [(-12, 1), (-308, 300), (-323, -300)])
@pytest.mark.parametrize("top", [7, 20, 48])
def test_div(lib, lo, hi, top):
    rng = np.random.default_rng(top)
    n = 400_000
    b = np.maximum(1, np.exp2(rng.uniform(0, top, n)).astype(np.int64)).astype(np.float64)
    a = 10.0 ** rng.uniform(lo, hi, n)
    assert bad(lib.div_bad, a, b) == 0
    # numerators whose quotients lie as near to a midpoint as the format allows:
    # a = RN(b (q + half a unit)) and its neighbours
    q = 1.0 + rng.integers(0, 1 << 52, n) * 2.0 ** -52
    for k in (-1, 0, 1):
        m = ((b.astype(np.longdouble) * (q.astype(np.longdouble) + np.longdouble(2.0) ** -53))
             .astype(np.float64).view(np.int64) + k).view(np.float64)
        assert bad(lib.div_bad, np.ascontiguousarray(m), b) == 0
    for x in (0.0, 1.0, 5e-324, 1.7e308):
        assert bad(lib.div_bad, np.full(n, x), b) == 0
