"""The two-step kernel of large FP32 lattices: the states of single steps, bit
for bit, at the edges of its strips of 56 columns (whole strips, one column
more, odd widths) and of its bands, for walls on each side, moving walls, both
periodic wraps, a force, both schemes and obstacles that touch every edge; the
buffer one step earlier that the diagnostics read."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flow(nx, ny, kind):
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    if kind in ("periodic", "periodic_mask"):
        wl = W.taylor_green(nx, ny, 0.8, 0.19, 0.02, u0=0.02, seed=1)
    elif kind == "force":
        wl = W.poiseuille(ny=ny, nx=nx, a=0.5, cs2=0.075, nu=0.02, U=0.02)
    elif kind == "side_walls":
        wl = W.cavity(nx, ny, 0.5, 0.075, 0.03, 100.0).with_(
            periodic_y=1, wall_u=((0.0, 0.01), (0.0, -0.02), (0.0, 0.0), (0.0, 0.0)))
    else:
        wl = W.cavity(nx, ny, 0.5, 0.075, 0.05, 400.0).with_(
            wall_u=((0.0, 0.01), (0.0, -0.02), (0.01, 0.0), (0.03, 0.0)))
    if kind.endswith("mask"):
        m = W.random_obstacles(nx, ny, seed=3, coverage=0.08)
        m[::5, 0] = m[::3, nx - 1] = 1
        m[0, ::7] = m[ny - 1, ::4] = 1
        wl = wl.with_(mask=m)
    return wl.with_(rho=r, ux=u, uy=v)


@pytest.mark.parametrize("kind", ["periodic", "force", "side_walls", "walls", "walls_mask",
                                  "periodic_mask"])
@pytest.mark.parametrize("nx,ny", [(504, 400), (505, 401), (3000, 67), (283, 709), (64, 3200)])
def test_two_step_kernel_matches_single_steps(nx, ny, kind):
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, kind)
    for scheme in (0, 1):
        a = Lattice.from_workload(wl, precision=32, scheme=scheme)
        b = Lattice.from_workload(wl, precision=32, scheme=scheme)
        launches = 0
        for n in (1, 2, 3, 8, 53):
            a.step(n)
            for _ in range(n):
                b.step(1)
            launches += n - max(0, (n - 1) // 2)
            assert np.array_equal(a.get_f(), b.get_f()), n
            # the step-to-step change and the residual read both buffers
            assert np.array_equal(a.diagnostics()[1], b.diagnostics()[1]), n
        # lattices with walls along x take the path from a width of 281 on
        assert a.launch_count == (67 if nx <= 280 and not wl.periodic_x else launches)
        assert a.step_count == b.step_count == b.launch_count == 67
        a.close()
        b.close()


def test_no_collision_takes_single_steps():
    """The streaming-only mode has no two-step form."""
    from paper_2103_02119_gb300.lbm import Lattice
    g = Lattice(512, 512, 0.5, 0.075, [1.0] * 9, precision=32, scheme=-1)
    g.step(9)
    assert g.launch_count == 9
    g.close()
