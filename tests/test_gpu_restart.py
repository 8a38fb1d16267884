"""Restart from a saved state, bit for bit: a run that is read out, set again
and continued equals the uninterrupted run, in 2-D binary64 on every compiled
lattice and on grids of each launch shape (16 x 8 and 16 x 16 tiles, one and
two CTAs per SM), and in 1-D on both sides of the short-problem kernels'
limit."""
import numpy as np
import pytest

from paper_1909_08390_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def restart_equals_run(kw, states, split, nsteps, at):
    from paper_1909_08390_gb300 import fdlb as F
    with F.Solver(**kw) as a, F.Solver(**kw) as b:
        for s in (a, b):
            s.init_riemann(states, *split)
        a.step(nsteps)
        b.step(at)
        b.set_state(b.state())
        b.step(nsteps - at)
        assert np.array_equal(a.state(), b.state())


@pytest.mark.parametrize("Q", [(8, 8), (5, 3), (3, 3)])
@pytest.mark.parametrize("shape", [(37, 29), (192, 187), (400, 304)])
def test_2d_binary64_restart_is_bitwise(shape, Q):
    nx, ny = shape
    restart_equals_run(dict(d=2, nx=nx, ny=ny, x0=0.0, x1=1.0, y0=0.0, y1=1.0, Qphi=Q[0], Qchi=Q[1],
                            gamma=1.4, tau=1e-5, dt=2e-4 * 64.0 / max(nx, ny, 64)),
                       W.C11_STATES, (0.5, 0.5), 7, 3)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("Q", [(8, 8), (5, 3), (3, 3)])
@pytest.mark.parametrize("nx", [400, 12001])
def test_1d_restart_is_bitwise(nx, Q, precision):
    restart_equals_run(dict(d=1, nx=nx, x0=-0.5, x1=0.5, Qphi=Q[0], Qchi=Q[1], gamma=1.4, tau=1e-5,
                            dt=0.02 / nx, precision=precision),
                       W.sod_1d().states, (0.0,), 7, 3)
