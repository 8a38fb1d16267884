"""The 2-D binary64 kernels' march on either side of its scaling: tiles whose
values are too small to scale (below 2^-823) march in binary64.  The step is
homogeneous of degree one in the populations, so a state times a power of two
gives the result times that power: both marches within the parity bar (1e-12)
of each other, and the same u and T.  And an invalid cell is reported."""
import numpy as np
import pytest

from paper_1909_08390_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("Q", [(8, 8), (5, 3)])
@pytest.mark.parametrize("shape", [(33, 17), (16, 16), (300, 270)])
def test_scaled_and_binary64_marches_agree(shape, Q, bc):
    from paper_1909_08390_gb300 import fdlb as F
    nx, ny = shape
    kw = dict(d=2, nx=nx, ny=ny, x0=0.0, x1=1.0, y0=0.0, y1=1.0, bc=bc, Qphi=Q[0], Qchi=Q[1],
              gamma=1.4, tau=1e-4, dt=2e-4 * 16.0 / max(nx, ny, 16))
    with F.Solver(**kw) as a, F.Solver(**kw) as b:
        F0 = W.smooth_random_populations(a.shape, seed=nx + bc, amp=0.3)
        a.set_state(F0)
        b.set_state(np.ldexp(F0, -840))
        a.step(4)
        b.step(4)
        G, H = a.state(), np.ldexp(b.state(), 840)
        assert np.abs(G - H).max() < 1e-12 * np.abs(G).max()
        for m, k in ((1, 1.0), (3, 0.0)):
            x, y = a.moments()[m], b.moments()[m]
            assert np.abs(x - y).max() < 1e-12 * max(np.abs(x).max(), k)


@pytest.mark.parametrize("value", [np.nan, np.inf, -1e3])
def test_an_invalid_cell_is_reported(value):
    from paper_1909_08390_gb300 import fdlb as F
    with F.Solver(d=2, nx=40, ny=24, x0=0.0, x1=1.0, y0=0.0, y1=1.0, tau=1e-4, dt=2e-4) as s:
        F0 = W.smooth_random_populations(s.shape, seed=1, amp=0.1)
        s.set_state(F0)
        s.step(1)
        F0[:, 7, 11] = value
        s.set_state(F0)
        with pytest.raises(F.FdlbError) as e:
            s.step(1)
        assert e.value.code == F.FDLB_EUNSTABLE
