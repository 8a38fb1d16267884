"""The memory layout of mixed 2-D contexts: populations padded to whole 16-cell
tiles, or not where a grid is too thin for it.  The state exchange is exact in
both, and a run agrees with the binary64 one to the mixed path's bar (1e-5,
a few steps) on grids whose last tiles are ragged, both boundaries."""
import numpy as np
import pytest

from paper_1909_08390_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("Q", [(8, 8), (5, 3)])
@pytest.mark.parametrize("shape", [(33, 17), (36, 31), (15, 16), (2, 40000), (40001, 3)])
def test_padded_and_thin_grids(shape, Q, bc):
    from paper_1909_08390_gb300 import fdlb as F
    nx, ny = shape
    kw = dict(d=2, nx=nx, ny=ny, x0=0.0, x1=1.0, y0=0.0, y1=1.0, bc=bc, Qphi=Q[0], Qchi=Q[1],
              gamma=1.4, tau=1e-5, dt=0.1 / (max(nx, ny) * 4.2))
    with F.Solver(**kw, precision=F.FDLB_MIXED) as m, F.Solver(**kw) as d:
        F0 = W.smooth_random_populations(m.shape, seed=nx + ny + bc, amp=0.2).astype(np.float32)
        F0 = F0.astype(np.float64) * (1.0 + 2.0 ** -30)  # pairs hold it exactly
        m.set_state(F0)
        assert np.array_equal(m.state(), F0)
        d.set_state(F0)
        m.step(3)
        d.step(3)
        for a, b, floor in zip(m.moments(), d.moments(), (0.0, 1.0, 1.0, 0.0)):
            assert np.abs(a - b).max() < 1e-5 * max(np.abs(b).max(), floor)
