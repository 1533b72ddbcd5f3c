"""The integer stencil arithmetic (csrc/stencil_fixed.cuh, plain C++) on the
host: position between nodes against exact integers, weights against Eq. 14 in
50 digits."""
import ctypes as C
import math
import os
import shutil
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2102_01305_gb300.build import CSRC

mp = pytest.importorskip("mpmath").mp


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("stencil")
    src, out = os.path.join(d, "s.cpp"), os.path.join(d, "s.so")
    with open(src, "w") as f:
        f.write('#include "stencil_fixed.cuh"\n'
                'extern "C" int split(unsigned long long b, long long* o) { return ibl::split_bits(b, o[0], o[1]); }\n'
                'extern "C" void weights(long long t, long long* w) { ibl::fixed_weights(t, *(long long(*)[4])w); }\n')
    subprocess.run([cxx, "-O2", "-shared", "-fPIC", "-I", CSRC, src, "-o", out], check=True)
    so = C.CDLL(out)
    so.split.argtypes = [C.c_ulonglong, C.c_void_p]
    so.weights.argtypes = [C.c_longlong, C.c_void_p]
    so.weights.restype = None
    return so


def _split(lib, x):
    o = (C.c_longlong * 2)()
    ok = lib.split(struct.unpack("<Q", struct.pack("<d", x))[0], o)
    return ok, o[0], o[1]


def _coordinates():
    rng = np.random.default_rng(2)
    xs = [0.0, -0.0, 0.5, -0.5, 1.0, -1.0, 3.0, -7.0, 255.999999, math.nextafter(3.0, 0.0), math.nextafter(-3.0, -9.0),
          5e-324, -5e-324, 1e-20, -1e-20, -2.0 ** -64, -2.0 ** -65, 2.0 ** -64, -1e-19, 2.0 ** 31 - 0.25, -2.0 ** 31 + 0.25,
          2.0 ** -1022, -2.0 ** -1022]
    xs += list(rng.uniform(-400, 400, size=3000)) + list(np.ldexp(rng.uniform(-1, 1, size=3000), rng.integers(-80, 31, size=3000)))
    return [float(x) for x in xs]


def test_split(lib):
    for x in _coordinates():
        ok, fl, t = _split(lib, x)
        exact = Fraction(x)
        assert ok
        if -Fraction(1, 2 ** 64) < exact < 0:
            assert (fl, t) == (0, -2 ** 63)
        else:
            assert fl == math.floor(x)
            # t / 2^64 + 1/2 is the fraction, less than one unit off
            assert abs(Fraction(t, 2 ** 64) + Fraction(1, 2) - (exact - fl)) < Fraction(1, 2 ** 64)
    for x in (2.0 ** 31, -2.0 ** 31, 1e300, math.inf, -math.inf, math.nan):
        assert not _split(lib, x)[0]


def test_weights(lib):
    mp.dps = 50
    rng = np.random.default_rng(4)
    ts = [-2 ** 63, -2 ** 63 + 1, -1, 0, 1, 2 ** 63 - 1, -2 ** 62, 2 ** 62, -2 ** 63 + 2 ** 20]
    ts += [int(v) for v in rng.integers(-2 ** 63, 2 ** 63 - 1, size=20000)]
    ts += [int(-2 ** 63 + 2 ** k) for k in range(60)] + [int(2 ** 63 - 2 ** k) for k in range(60)]
    w = (C.c_longlong * 4)()
    worst = 0
    for t in ts:
        lib.weights(t, w)
        s = mp.mpf(t) / 2 ** 64 + mp.mpf(1) / 2
        for k in range(4):
            exact = (1 + mp.cos(mp.pi / 2 * (s - (k - 1)))) / 4
            worst = max(worst, abs(w[k] - exact * 2 ** 60))
            assert 0 <= w[k] <= 2 ** 59
        assert w[0] + w[2] == w[1] + w[3] == 2 ** 59
    assert worst <= 1
    lib.weights(-2 ** 63, w)
    assert list(w) == [2 ** 58, 2 ** 59, 2 ** 58, 0]
