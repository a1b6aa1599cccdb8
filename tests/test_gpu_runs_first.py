"""FP32 lattices of 80,000 to 200,000 cells that the many-step kernel cannot take: which
of the row-band kernel's runs and the two-step kernel steps them (by the number of
launches), and the states."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STILL = ((0.0, 0.0),) * 4
WALLS = {"rest": STILL, "lid": STILL[:3] + ((0.03, 0.0),), "sides": ((0.0, 0.01), (0.0, -0.02)) + STILL[:2]}

TWO, FIRST, BAND = 31, 56, 60     # launches of a call of 60: two steps each; 50, then those; one each


@pytest.mark.parametrize("nx,ny,px,walls,masked,launches", [
    (900, 90, 0, "rest", False, FIRST), (900, 90, 0, "lid", False, FIRST), (900, 90, 0, "sides", False, BAND),
    (900, 90, 0, "rest", True, TWO), (900, 90, 0, "lid", True, TWO), (900, 90, 0, "sides", True, FIRST),
    (900, 90, 1, "rest", False, TWO), (901, 90, 1, "rest", False, FIRST), (900, 90, 1, "lid", False, FIRST),
    (900, 90, 1, "lid", True, TWO), (900, 206, 0, "rest", False, TWO), (900, 206, 0, "sides", False, FIRST),
    (900, 223, 0, "sides", False, TWO)])
def test_route_and_states(nx, ny, px, walls, masked, launches):
    from paper_2103_02119_gb300.lbm import Lattice
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    wl = W.cavity(nx, ny, 0.5, 0.075, 0.05, 400.0).with_(rho=r, ux=u, uy=v, periodic_x=px, wall_u=WALLS[walls])
    if masked:
        wl = wl.with_(mask=W.random_obstacles(nx, ny, seed=3, coverage=0.05))
    a, b = (Lattice.from_workload(wl, precision=32) for _ in range(2))
    a.step(60)
    assert a.launch_count == launches
    for n in (1, 20, 103, 2):
        a.step(n)
    for _ in range(186):
        b.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    assert np.array_equal(a.diagnostics()[1], b.diagnostics()[1])
    a.close()
    b.close()
