"""The 2-D binary64 kernels on tiles whose values span many binades: a smooth
density with a jump by up to 1e17 inside a tile.  Small cells beside large ones
keep their own digits: n and T of every cell are compared relative to that
cell's value (u to 1, with T of order one), with the same run marched in
binary64 (the state times 2^-840, which the fixed-point march does not take;
the step is homogeneous of degree one), and n with the oracle on the cells the
jump's windows don't reach.

Tolerance.  Where the fixed-point march runs, a cell lies at most 16 times
below the largest value its line reads, so a flux difference is within 62 units
of 2^-59 of 32 times the cell's value (the power of two above the largest):
3.5e-15.  The binary64 march's own error is below 64 rounding units of it,
0.7e-14.  Three
stages with two axes, each times dt |p| / ds < 0.1 and relaxed (u and T lose
up to another factor of 10 to the moments' cancellations): 1e-13 for n, 1e-12
for u and T, in place of which the march on one scale for all cells loses
5e-14 (jump of 1e4) to all digits (1e17) of a cell's flux differences."""
import numpy as np
import pytest

from paper_1909_08390_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def fields(nx, ny, jump, axis):
    x = (np.arange(nx) + 0.5)[None, :] + np.zeros((ny, 1))
    y = (np.arange(ny) + 0.5)[:, None] + np.zeros((1, nx))
    s = x if axis == 0 else y
    n = np.where(s < 23, 1.0, 1.0 / jump) * (1.0 + 0.1 * np.sin(x / 5.0 + 1.0) * np.cos(y / 7.0))
    u = 0.1 * np.sin(x / 9.0 + 0.3 * y / 7.0)
    v = 0.1 * np.cos(y / 8.0 - 0.2 * x / 7.0)
    T = 1.0 + 0.1 * np.sin(x / 6.0 + y / 6.0)
    return n, u, v, T


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("Q", [(8, 8), (5, 3)])
@pytest.mark.parametrize("jump", [1e2, 1e4, 1e6, 1e8, 1e17])
def test_small_cells_keep_their_digits(oracle, jump, Q, axis):
    from paper_1909_08390_gb300 import fdlb as F
    nx, ny = 60, 52
    kw = dict(d=2, nx=nx, ny=ny, x0=0.0, x1=float(nx), y0=0.0, y1=float(ny), Qphi=Q[0], Qchi=Q[1],
              gamma=1.4, tau=0.05, dt=0.02)
    pr = oracle.Problem(**kw)
    F0 = oracle.init_fields(pr, *fields(nx, ny, jump, axis))
    with F.Solver(**kw) as a, F.Solver(**kw) as b:
        a.set_state(F0)
        b.set_state(np.ldexp(F0, -840))
        a.step(1)
        b.step(1)
        (n, u, v, T), (m, w, z, S) = a.moments(), b.moments()
    m = np.ldexp(m, 840)
    on = oracle.moments(pr, oracle.step(pr, F0, 1))[0]
    cells = np.arange(nx)[None, :] if axis == 0 else np.arange(ny)[:, None]
    far = np.broadcast_to(np.abs(cells + 0.5 - 23) > 16, n.shape)
    print("n %.1e u %.1e v %.1e T %.1e, n against the oracle %.1e" % (
        np.abs(n / m - 1).max(), np.abs(u - w).max(), np.abs(v - z).max(), np.abs(T / S - 1).max(),
        np.abs(n / on - 1)[far].max()))
    assert np.abs(n / m - 1).max() < 1e-13
    assert np.abs(n / on - 1)[far].max() < 1e-13
    assert max(np.abs(u - w).max(), np.abs(v - z).max(), np.abs(T / S - 1).max()) < 1e-12
