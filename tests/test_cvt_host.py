"""The integer binary32 <-> binary64 conversions (fdlb_cvt.cuh), compiled for
the host: the bits of the machine's conversions on values around every edge
(zeros, denormals, halfway cases, the largest values, infinities, NaN)."""
import ctypes
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host", "cvt_host.cpp")
LIB = os.path.join(HERE, "host", "_build", "libcvthost.so")


def _lib():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    subprocess.run(["g++", "-std=c++17", "-O2", "-fPIC", "-shared", SRC, "-o", LIB], check=True)
    L = ctypes.CDLL(LIB)
    for f in (L.widen_all, L.narrow_all):
        f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]
    return L


def test_conversions_give_the_machines_bits():
    L = _lib()
    rng = np.random.default_rng(0)
    b = rng.integers(0, 2 ** 32, 400000, dtype=np.uint32)
    b[:1000] = np.concatenate([np.arange(250), 0x7f800000 - 125 + np.arange(250), 0x00800000 - 125 + np.arange(250),
                               0x80000000 + np.arange(250)]).astype(np.uint32)
    x = b.view(np.float32)
    y = np.empty(x.size)
    L.widen_all(x.ctypes.data, y.ctypes.data, x.size)
    with np.errstate(all="ignore"):
        want = x.astype(np.float64)
        ok = ~np.isnan(x)
        assert np.array_equal(y.view(np.uint64)[ok], want.view(np.uint64)[ok]) and np.all(np.isnan(y[~ok]))
        # halfway and one binary64 unit around it, the edges of the normal range, anything
        h = want[ok][np.isfinite(want[ok])]
        nxt = np.nextafter(h.astype(np.float32), np.float32(np.inf)).astype(np.float64)
        mid = h + (nxt - h) / 2
        v = np.concatenate([h, mid, np.nextafter(mid, np.inf), np.nextafter(mid, -np.inf),
                            rng.integers(0, 2 ** 64, 200000, dtype=np.uint64).view(np.float64),
                            rng.normal(size=100000) * 2.0 ** rng.integers(-160, 140, 100000),
                            [0.0, -0.0, np.inf, -np.inf, 3.4028235677973366e38, 3.4028235677973362e38, 2.0 ** -126,
                             np.nextafter(2.0 ** -126, 0)]])
        z = np.empty(v.size, np.float32)
        L.narrow_all(v.ctypes.data, z.ctypes.data, v.size)
        want = v.astype(np.float32)
    ok = ~np.isnan(v)
    assert np.array_equal(z.view(np.uint32)[ok], want.view(np.uint32)[ok]) and np.all(np.isnan(z[~ok]))
