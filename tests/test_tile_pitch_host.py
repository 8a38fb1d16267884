"""Mixed 2-D arrays padded to whole 16-cell tiles (csrc/fdlb_tile.cuh, compiled
for the host): every staged cell of every tile reads the cell or ghost source
it needs and never the padding, and the padding's size keeps its bound."""
import ctypes
import os
import subprocess

import pytest

import test_tile_index_host as T

SRC = os.path.join(T.HERE, "host", "tile_pitch_host.cpp")
LIB = os.path.join(T.HERE, "host", "_build", "libtilepitch.so")


@pytest.fixture(scope="module")
def lib():
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    if not os.path.exists(LIB) or os.path.getmtime(LIB) < max(map(os.path.getmtime, (SRC, T.SRC, T.HDR))):
        tmp = LIB + f".{os.getpid()}"
        subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", SRC, "-o", tmp], check=True)
        os.replace(tmp, LIB)
    L = ctypes.CDLL(LIB)
    L.check_padded_chunks.argtypes = [ctypes.c_int] * 3
    L.pads.argtypes = [ctypes.c_longlong] * 2
    return L


@pytest.mark.parametrize("bc", [0, 1])
def test_padded_rows_read_the_right_cells(lib, bc):
    # periodic grids land chunks where their rows hold a multiple of 4 cells
    for nx in [n for n in list(range(1, 38)) + [47, 49, 63, 64, 66, 95] if bc == 0 or n % 4 == 0]:
        for ny in (1, 3, 5, 15, 16, 17, 33, 37):
            assert lib.check_padded_chunks(nx, ny, bc) == 0, (nx, ny, bc)


def test_padding_is_bounded(lib):
    """At most an eighth or 2^15 cells more, or twice the cells on grids of up
    to 2^18 cells so padded; near-square grids are always padded."""
    sides = [1, 2, 3, 5, 8, 15, 16, 17, 20, 31, 33, 64, 100, 127, 129, 200, 333, 400, 517, 640, 1000,
             2047, 2049, 4095, 16384, 40000]
    for nx in sides:
        for ny in sides:
            n, padded = nx * ny, -(-nx // 16) * 16 * (-(-ny // 16) * 16)
            if lib.pads(nx, ny):
                assert padded - n <= max(n // 8, 2 ** 15) or (padded <= 2 ** 18 and padded <= 2 * n), (nx, ny)
            elif min(nx, ny) * 4 > max(nx, ny):
                assert False, (nx, ny)
    assert not lib.pads(2, 16384) and not lib.pads(16384, 2) and lib.pads(512, 512) and lib.pads(2, 300)
