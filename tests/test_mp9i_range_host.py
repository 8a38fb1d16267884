"""Which lines the 2-D binary64 kernels march in fixed point (fdlb_mp9i.cuh),
compiled for the host: half lines of 8 cells down to a factor of 16 below the
largest of the 17 values read.  Against Sec. IV's formulas in exact rational
arithmetic, every cell whose stencil holds values of its own size keeps its
digits, whatever lies in the rest of the line.

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
    L.q_value.argtypes, L.q_value.restype = [ctypes.c_int64, ctypes.c_int], ctypes.c_double
    L.adv_two_scales.restype = L.adv_fp64.restype = ctypes.c_double
    L.adv_two_scales.argtypes = [ctypes.c_double] * 2 + [ctypes.c_int64, ctypes.c_int] * 2
    L.adv_fp64.argtypes = L.adv_two_scales.argtypes
    L.mp9_delta64.argtypes = [dp, ctypes.c_int, ctypes.c_int, dp]
    return L


def test_conversion_rounds_to_nearest(lib):
    """An integer goes back to binary64 within half a unit of its last place."""
    rng = np.random.default_rng(5)
    for k in range(4000):
        u = int(rng.integers(0, 2 ** 62)) >> int(rng.integers(0, 62))
        u = [u, -u, 2 ** 53 + 1, 2 ** 62 - 1, -1, 0][k % 6]
        got, want = Fr(lib.q_value(u, 1081)), Fr(u)
        last = Fr(2) ** max(abs(u).bit_length() - 53, 0)
        assert abs(got - want) <= last / 2, u


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
    """Half lines whose own cells lie at most 16 times below the largest value
    read march in fixed point, others in binary64; small values beside them
    don't matter."""
    rng = np.random.default_rng(1)
    base = rng.uniform(1.0, 1.9, 26)
    # (cell of the extended line, factor it is divided by, halves in fixed point
    # marching up and marching down); marching up the halves read cells 0-16 and
    # 8-24 for their own 5-12 and 13-20, marching down 1-17 and 9-25
    for i, ratio, up, down in ((8, 12.0, 3, 3), (8, 40.0, 2, 2), (20, 40.0, 1, 1), (21, 40.0, 3, 3), (2, 1e9, 3, 3),
                               (10, np.inf, 2, 2), (0, 1 / 40.0, 2, 3), (25, 1 / 40.0, 3, 1), (15, 1 / 40.0, 0, 0),
                               (4, 1 / 40.0, 2, 2), (23, 1 / 40.0, 1, 1)):
        ext = base.copy()
        ext[i] /= ratio
        for sgn, want in ((1, up), (-1, down)):
            took, got = march(lib, ext, sgn)
            assert took == want, (i, ratio, sgn)
            ref = np.zeros(16)
            lib.mp9_delta64(M._p(ext), 16, sgn, M._p(ref))
            for h in range(2):
                if not want >> h & 1:
                    assert np.array_equal(got[8 * h:8 * h + 8], ref[8 * h:8 * h + 8])
    for bad in (np.inf, np.nan, 2.0 ** 1010):
        ext = base.copy()
        ext[12] = bad
        assert march(lib, ext, 1)[0] == 0
    assert march(lib, np.zeros(26), 1)[0] == 0 and march(lib, base * 2.0 ** -900, 1)[0] == 0


def test_advection_term_of_two_scales(lib):
    """Flux differences on scales up to 2^8 apart add up within 4 units of the
    larger scale (one more than on one scale: the shift's), each coefficient's
    2^-60 and the conversion's rounding; with binary64 bits on one axis, within
    the roundings of the sum and of the conversions."""
    rng = np.random.default_rng(8)
    for i in range(3000):
        cx, cy = (float(x) for x in rng.choice([1.0, 0.013, 0.3, -0.7, 0.0], 2) * rng.uniform(0.5, 1, 2))
        ex, ey = 1081, 1081 - int(rng.integers(0, 9))
        if i % 2:
            ex, ey = ey, ex
        m = 2 ** int(rng.integers(1, 62))
        dx, dy = (int(rng.uniform(-1, 1) * m) for _ in range(2))
        sx, sy = Fr(2) ** (ex - 1081), Fr(2) ** (ey - 1081)
        want = abs(Fr(cx)) * dx * sx + abs(Fr(cy)) * dy * sy
        size = abs(Fr(cx)) * abs(dx) * sx + abs(Fr(cy)) * abs(dy) * sy
        big = max(abs(cx), abs(cy))
        unit = Fr(2) ** (int(np.frexp(big)[1]) + 3) if big else Fr(0)
        lost = Fr(big) * (abs(dx) * sx + abs(dy) * sy) / 2 ** 60
        got = Fr(lib.adv_two_scales(cx, cy, dx, ex, dy, ey))
        assert abs(got - want) <= 4 * unit + lost + abs(want) / 2 ** 53, (cx, cy, dx, ex, dy, ey)
        bits = int(np.array(float(dx) * float(sx)).view(np.int64))
        got = Fr(lib.adv_fp64(cx, cy, bits, 0, dy, ey))
        assert abs(got - want) <= 4 * size / 2 ** 53, (cx, cy, dx, ex, dy, ey)
