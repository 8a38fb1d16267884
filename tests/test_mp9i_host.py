"""The fixed-point MP-9 march of the binary64 stage kernels (fdlb_mp9i.cuh),
compiled for the host, against Sec. IV's formulas in exact rational
arithmetic, and beside the binary64 march.

Tolerance.  A unit is 2^-59 of the power of two above the line's largest
value.  Truncating the inputs moves a difference by at most 2 units and a
curvature by 4; the stencil's offset then moves by at most 2.6 units plus 3 of
its own rounding, 4 m - M by 20, and the bounds by at most 4/3 of that plus 3:
30 units.  The clamp moves by no more than what it clamps, so a flux
difference (two offsets and one difference) is within 62 units, and its
conversion truncates 2^-52 of itself.
"""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "host", "mp9i_host.cpp")
CSRC = os.path.join(os.path.dirname(HERE), "paper_1909_08390_gb300", "csrc")
HDRS = [os.path.join(CSRC, h) for h in ("fdlb_mp9.cuh", "fdlb_mp9i.cuh")]
LIB = os.path.join(HERE, "host", "_build", "libmp9ihost.so")


@pytest.fixture(scope="module")
def lib():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    if not os.path.exists(LIB) or os.path.getmtime(LIB) < max(map(os.path.getmtime, [SRC] + HDRS)):
        tmp = LIB + f".{os.getpid()}"
        subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", SRC,
                        "-o", tmp], check=True)
        os.replace(tmp, LIB)
    L = ctypes.CDLL(LIB)
    dp = ctypes.POINTER(ctypes.c_double)
    L.mp9i_line.argtypes = [dp, ctypes.c_int, ctypes.c_int, ctypes.c_int, dp]
    L.adv_term.argtypes = [ctypes.c_double] * 2 + [ctypes.c_int64] * 2 + [ctypes.c_int]
    L.adv_term.restype = ctypes.c_double
    L.mp9_delta64.argtypes = [dp, ctypes.c_int, ctypes.c_int, dp]
    return L


def _p(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def minmod4(a, b):
    xs = (4 * a - b, 4 * b - a, a, b)
    if all(x > 0 for x in xs) or all(x < 0 for x in xs):
        return min(xs, key=abs)
    return Fr(0)


def face(v):
    """Sec. IV literally: F^L, kept when it lies between F_s and F^MP, else
    clamped to [F^min, F^max]."""
    d = [v[k + 1] - v[k] for k in range(8)]
    a = Fr(sum(c * x for c, x in zip((-4, 37, -162, 479, 1120, -255, 50, -5), d)), 2520)
    cm, c0, c1 = d[3] - d[2], d[4] - d[3], d[5] - d[4]
    ul, md = 4 * d[3], (d[4] - minmod4(c0, c1)) / 2
    lc = d[3] / 2 + Fr(4, 3) * minmod4(cm, c0)
    lo = max(min(0, d[4], md), min(0, ul, lc))
    hi = min(max(0, d[4], md), max(0, ul, lc))
    return v[4] + min(max(a, lo), hi)


def flux_differences(ext, n, sgn):
    f = []
    for i in range(n + 1):
        s = (i - 1 if sgn > 0 else i) + 5
        f.append(face([Fr(float(ext[s + sgn * (j - 4)])) for j in range(9)]))
    return [sgn * (b - a) for a, b in zip(f, f[1:])]


def lines(rng, n):
    x = np.arange(n + 10.0)
    yield rng.uniform(0.5, 1.5, n + 10)
    yield rng.normal(size=n + 10)
    yield 2.0 + np.cumsum(rng.normal(size=n + 10)) * 0.01
    yield np.where(x < n / 2 + 3, 1.0, 1e-4) * (1 + 1e-3 * rng.normal(size=n + 10))
    yield 1.0 + 1e-13 * rng.normal(size=n + 10)
    yield np.full(n + 10, 0.3)
    yield 1.0 + 0.1 * np.sin(x / 3.0)
    yield rng.integers(-3, 4, n + 10).astype(float)
    yield np.where(rng.random(n + 10) < 0.3, 0.0, rng.normal(size=n + 10) * 1e-250)
    yield rng.uniform(-1, 1, n + 10) * 2.0 ** rng.integers(900, 1000, n + 10)
    yield np.concatenate([np.full(5, -0.0), rng.normal(size=n) * 1e3, np.zeros(5)])


@pytest.mark.parametrize("nc", [2, 4, 8, 16])
@pytest.mark.parametrize("sgn", [1, -1])
def test_march_matches_exact_flux_differences(lib, nc, sgn):
    rng = np.random.default_rng(10 * nc + sgn)
    worst = 0.0
    for _ in range(4):
        for ext in lines(rng, 16):
            ext = np.ascontiguousarray(ext)
            got, ref = np.zeros(16), np.zeros(16)
            emax = lib.mp9i_line(_p(ext), 16, sgn, nc, _p(got))
            lib.mp9_delta64(_p(ext), 16, sgn, _p(ref))
            unit = Fr(2) ** (emax - 1022 - 59)
            for g, b, w in zip(got, ref, flux_differences(ext, 16, sgn)):
                err = abs(Fr(float(g)) - w)
                assert err <= 62 * unit + abs(w) / 2 ** 52, (ext, float(g), float(w))
                # the binary64 march of the same line: a rounding unit of the
                # largest value per interface
                assert abs(Fr(float(b)) - w) <= 64 * 16 * unit
                worst = max(worst, float(err / unit) if abs(w) < 2 ** 52 * unit else 0.0)
    print(f"largest error {worst:.1f} units (below 2^52 units)")


def test_march_is_the_same_whatever_its_segments(lib):
    """On one scale the flux differences are integers: 2-, 4-, 8- and 16-cell
    segments give the same bits."""
    rng = np.random.default_rng(3)
    for ext in lines(rng, 16):
        ext = np.ascontiguousarray(ext)
        for sgn in (1, -1):
            got = []
            for nc in (2, 4, 8, 16):
                o = np.zeros(16)
                lib.mp9i_line(_p(ext), 16, sgn, nc, _p(o))
                got.append(o.copy())
            assert all(np.array_equal(got[0], o) for o in got[1:])


def test_advection_term_matches_rational_arithmetic(lib):
    """|cx| dx + |cy| dy from 61-bit coefficients: 3 units of the product's
    scale (the coefficient's power of two over 8), then the conversion's
    truncation; a coefficient loses at most 2^-61 of the larger one."""
    rng = np.random.default_rng(7)
    top = 5 * 2 ** 60  # flux differences stay below 2^62.4
    for i in range(3000):
        cx, cy = (float(x) for x in rng.choice([1.0, 0.013, 2.0 ** -40, 0.3, -0.7, 0.0, 1e-30], 2) * rng.uniform(0.5, 1, 2))
        m = 2 ** int(rng.integers(1, 63))
        dx, dy = (int(np.clip(int(rng.uniform(-1, 1) * m), -top, top)) for _ in range(2))
        if i % 3 == 0:
            dx, dy = [(top, top), (-top, -top), (0, -1)][i // 3 % 3]
        big = max(abs(cx), abs(cy))
        got = Fr(lib.adv_term(cx, cy, dx, dy, 1081))
        want = abs(Fr(cx)) * dx + abs(Fr(cy)) * dy
        unit = Fr(2) ** (int(np.frexp(big)[1]) + 3) if big else Fr(0)
        lost = Fr(big) * (abs(dx) + abs(dy)) / 2 ** 60
        assert abs(got - want) <= 3 * unit + lost + abs(want) / 2 ** 52, (cx, cy, dx, dy)
