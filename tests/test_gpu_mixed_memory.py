"""A mixed context of a thin 2-D grid takes about the memory of its own cells:
eleven binary32 arrays of P populations and nine binary64 fields, not those of
a grid rounded up to whole tiles."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 16384), (16384, 2), (400, 400)])
def test_memory_of_mixed_grids(shape):
    import torch
    from paper_1909_08390_gb300 import fdlb as F
    nx, ny = shape
    torch.cuda.init()
    with F.Solver(d=2, nx=32, ny=32, precision=F.FDLB_MIXED):  # the library's own memory
        pass
    before = torch.cuda.mem_get_info()[0]
    with F.Solver(d=2, nx=nx, ny=ny, x0=0.0, x1=1.0, y0=0.0, y1=1.0, tau=1e-5, dt=1e-6,
                  precision=F.FDLB_MIXED) as s:
        used = before - torch.cuda.mem_get_info()[0]
        own = nx * ny * (s.P * 11 * 4 + 9 * 8)
    assert used < 1.2 * own + (8 << 20), (used, own)
