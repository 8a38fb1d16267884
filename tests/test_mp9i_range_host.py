"""Which tiles the 2-D binary64 kernels march in fixed point (fdlb_mp9i.cuh),
compiled for the host: own cells down to a factor of 16 below the largest value
of tile and halo.  Against Sec. IV's formulas in exact rational arithmetic,
every cell whose stencil holds values of its own size keeps its digits,
whatever lies in the rest of the tile.

Tolerance.  In fixed point a flux difference is within 62 units (the bound of
the march's own test), a unit is 2^-59 of the power of two above the largest
value, and that is at most 2 * 17 times the cell's: 62 * 34 * 2^-59 < 2^-47.9 of
it.  In binary64 it is within 64 rounding units of the stencil's largest value,
here at most 4 times the cell's: 2^-45."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

import test_mp9i_host as M

SRC = os.path.join(M.HERE, "host", "mp9i_range_host.cpp")
LIB = os.path.join(M.HERE, "host", "_build", "libmp9irange.so")


@pytest.fixture(scope="module")
def lib():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    if not os.path.exists(LIB) or os.path.getmtime(LIB) < max(map(os.path.getmtime, [SRC, M.SRC] + M.HDRS)):
        tmp = LIB + f".{os.getpid()}"
        subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", SRC,
                        "-o", tmp], check=True)
        os.replace(tmp, LIB)
    L = ctypes.CDLL(LIB)
    dp = ctypes.POINTER(ctypes.c_double)
    L.mp9i_choice.argtypes = [dp, ctypes.c_int, dp]
    L.mp9_delta64.argtypes = [dp, ctypes.c_int, ctypes.c_int, dp]
    return L


def march(lib, ext, sgn):
    ext = np.ascontiguousarray(ext)
    out = np.zeros(16)
    return lib.mp9i_choice(M._p(ext), sgn, M._p(out)), out


@pytest.mark.parametrize("jump", [1.0, 4.0, 12.0, 1e2, 1e4, 1e6, 1e8, 1e17])
@pytest.mark.parametrize("at", [3, 9, 13, 19, 23])
def test_cells_keep_their_digits(lib, jump, at):
    rng = np.random.default_rng(at)
    x = np.arange(26.0)
    for trial in range(6):
        low = np.where(x < at, 1.0, 1.0 / jump)
        ext = (low if trial % 2 else low[::-1]) * rng.uniform(0.5, 1.0)
        ext = ext * (1.0 + 0.1 * np.sin(x / rng.uniform(2, 6)) if trial < 4 else rng.uniform(1.0, 1.2, 26))
        for sgn in (1, -1):
            _, got = march(lib, ext, sgn)
            for c, w in enumerate(M.flux_differences(ext, 16, sgn)):
                own = abs(ext[c + 5])
                if np.abs(ext[c:c + 11]).max() <= 4 * own:
                    assert abs(Fr(float(got[c])) - w) <= Fr(float(own)) / 2 ** 45, (jump, at, c)


def test_where_the_line_lies(lib):
    """Own cells at most 16 times below the largest value march in fixed
    point, cells further below or zero in binary64; small cells of the halo
    alone don't matter."""
    rng = np.random.default_rng(1)
    base = rng.uniform(1.0, 1.9, 26)
    for i, ratio, fixed in ((8, 12.0, 1), (8, 40.0, 0), (20, 40.0, 0), (21, 40.0, 1), (2, 1e9, 1), (10, np.inf, 0)):
        ext = base.copy()
        ext[i] /= ratio
        took, got = march(lib, ext, 1)
        assert took == fixed, (i, ratio)
        if not fixed:
            want = np.zeros(16)
            lib.mp9_delta64(M._p(ext), 16, 1, M._p(want))
            assert np.array_equal(got, want)
    for bad in (np.inf, np.nan, 2.0 ** 1010):
        ext = base.copy()
        ext[3] = bad
        assert march(lib, ext, 1)[0] == 0
    assert march(lib, np.zeros(26), 1)[0] == 0 and march(lib, base * 2.0 ** -900, 1)[0] == 0
