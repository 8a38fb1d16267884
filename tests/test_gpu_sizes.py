"""Single problems on either side of every size at which the dispatch changes
its kernels: 1-D short-problem blocks, 31-, 63- and 127-cell tiles (binary64;
mixed also 15-cell tiles), 2-D binary64 grids with an SM for each 16 x 8
tile, for each 16 x 16 tile only, and for neither.

1-D results don't depend on the tiling: an outlet problem equals, bit for bit,
the same problem as the only member of a batch, and a periodic problem of
several periods equals the run of one period in each of them (the cell size is
a power of two, so both have the same constants).  2-D and one long periodic
1-D run are compared with the oracle within the parity bar, 1e-12."""
import numpy as np
import pytest

from paper_1909_08390_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (Q, precision, lengths): the last short problem, the first tiled one, the
# first length of each larger tile
LENGTHS = [((8, 8), 0, (4096, 4097, 9577, 19305)), ((5, 3), 0, (8192, 8193, 9577, 19305)),
           ((8, 8), 1, (4096, 4097, 4713, 9577, 19305)), ((5, 3), 1, (4096, 4097, 4713, 9577, 19305))]
CASES = [(Q, prec, nx) for Q, prec, lengths in LENGTHS for nx in lengths]
SHORT = [((5, 3), prec, nx) for prec in (0, 1) for nx in (1, 5, 130, 777, 3201)]


def periodic(nx, Q, precision):
    from paper_1909_08390_gb300 import fdlb as F
    return F.Solver(d=1, nx=nx, x0=0.0, x1=nx / 1024.0, bc=1, Qphi=Q[0], Qchi=Q[1], gamma=1.4,
                    tau=1e-5, dt=2e-5, precision=precision)


@pytest.mark.parametrize("Q,precision,nx", CASES + SHORT)
def test_outlet_run_equals_a_batch_of_one(Q, precision, nx):
    from paper_1909_08390_gb300 import fdlb as F
    st = np.array([W.sod_1d().states])
    kw = dict(tau=1e-6, dt=0.02 / max(nx, 100), precision=precision)
    with F.BatchSolver([nx], [1.4], Qphi=Q[0], Qchi=Q[1], **kw) as b:
        b.init_riemann(st, np.array([0.01]))
        b.step(19)
        got = b.state()
    with F.Solver(d=1, nx=nx, x0=-0.5, x1=0.5, Qphi=Q[0], Qchi=Q[1], gamma=1.4, **kw) as s:
        s.init_riemann(st[0], 0.01)
        s.step(19)
        assert np.array_equal(s.state(), got)


@pytest.mark.parametrize("Q,precision,nx", CASES)
def test_long_periodic_run_repeats_its_period(Q, precision, nx):
    period = max(p for p in range(1, 3000) if nx % p == 0)
    with periodic(period, Q, precision) as s:
        F0 = W.smooth_random_populations(s.shape, seed=nx, amp=0.3)
        s.set_state(F0)
        s.step(5)
        want = s.state()
    with periodic(nx, Q, precision) as s:
        s.set_state(np.tile(F0, nx // period))
        s.step(5)
        got = s.state()
    assert np.array_equal(got, np.tile(want, nx // period))


def test_long_periodic_run_against_the_oracle(oracle):
    pr = oracle.Problem(d=1, nx=9583, x0=0.0, x1=1.0, bc=1, Qphi=8, Qchi=8, gamma=1.4, tau=1e-5, dt=2e-6)
    from paper_1909_08390_gb300 import fdlb as F
    F0 = W.smooth_random_populations(pr.shape, seed=9, amp=0.3)
    want = oracle.step(pr, F0, 4)
    with F.Solver(d=1, nx=pr.nx, x0=0.0, x1=1.0, bc=1, gamma=1.4, tau=1e-5, dt=2e-6) as s:
        s.set_state(F0)
        s.step(4)
        assert np.abs(s.state() - want).max() < 1e-12 * np.abs(want).max()


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("Q", [(8, 8), (5, 3)])
@pytest.mark.parametrize("shape", [(192, 187), (187, 192), (230, 210)])
def test_2d_binary64_grids_of_each_launch_shape(oracle, shape, Q, bc):
    from paper_1909_08390_gb300 import fdlb as F
    nx, ny = shape
    kw = dict(d=2, nx=nx, ny=ny, x0=0.0, x1=1.0, y0=0.0, y1=1.0, bc=bc, Qphi=Q[0], Qchi=Q[1],
              gamma=1.4, tau=1e-4, dt=1e-5)
    pr = oracle.Problem(**kw)
    F0 = W.smooth_random_populations(pr.shape, seed=nx + bc, amp=0.3)
    want = oracle.step(pr, F0, 2)
    with F.Solver(**kw) as s:
        s.set_state(F0)
        s.step(2)
        assert np.abs(s.state() - want).max() < 1e-12 * np.abs(want).max()
