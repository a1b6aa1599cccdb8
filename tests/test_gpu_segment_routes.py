"""FP32 lattices of one segment of the row-band kernel between walls: whether its runs
or the two-step kernel step them (by the number of launches), and the states."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STILL = ((0.0, 0.0),) * 4
LID = STILL[:3] + ((0.03, 0.0),)
TWO, FIRST = 31, 56               # launches of a call of 60: two steps each; 50, then those


@pytest.mark.parametrize("nx,ny,px,walls,masked,launches", [
    (169, 3551, 0, STILL, False, FIRST), (184, 3260, 0, STILL, False, FIRST), (192, 3125, 0, STILL, False, FIRST),
    (225, 2667, 0, STILL, False, FIRST), (232, 2586, 0, STILL, False, FIRST), (256, 5859, 0, STILL, False, FIRST),
    (168, 3572, 0, STILL, False, TWO), (193, 3109, 0, STILL, False, TWO), (224, 2679, 0, STILL, False, TWO),
    (257, 2335, 0, STILL, False, TWO), (128, 4688, 0, STILL, False, TWO), (184, 2608, 0, STILL, False, TWO),
    (184, 8153, 0, STILL, False, TWO), (184, 3260, 1, STILL, False, TWO), (184, 3260, 0, LID, False, TWO),
    (184, 3260, 0, STILL, True, TWO)])
def test_route_and_states(nx, ny, px, walls, masked, launches):
    from paper_2103_02119_gb300.lbm import Lattice
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    wl = W.cavity(nx, ny, 0.5, 0.075, 0.05, 400.0).with_(rho=r, ux=u, uy=v, periodic_x=px, wall_u=walls)
    if masked:
        wl = wl.with_(mask=W.random_obstacles(nx, ny, seed=3, coverage=0.05))
    a, b = (Lattice.from_workload(wl, precision=32) for _ in range(2))
    a.step(60)
    assert a.launch_count == launches
    a.step(103)
    for _ in range(163):
        b.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close()
    b.close()
