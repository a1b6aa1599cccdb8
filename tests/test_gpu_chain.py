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
        assert a.launch_count == launches
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


@pytest.mark.parametrize("shapes", [[(64, 16), (65, 17)], [(64, 65), (65, 64), (260, 16), (261, 17)],
                                    [(505, 67), (283, 40), (112, 200), (113, 33), (64, 300)]])
def test_two_step_kernel_of_batches(shapes):
    """A batch whose lattices can all take two steps per launch (at least 64 by
    16 cells): the states of single-lattice steps bit for bit, with one launch
    for two steps; the residual from both buffers; a lattice that retires and
    comes back at the other parity; one that cannot take it (63 wide) sends the
    batch back to a launch per step."""
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    kinds = ["periodic", "force", "side_walls", "walls", "walls_mask", "periodic_mask"]
    ws = [_flow(nx, ny, k) for nx, ny in shapes for k in kinds]
    ws = [w if w.mask is not None else w.with_(mask=np.zeros((w.ny, w.nx), np.uint8)) for w in ws]
    schemes = [0 if i % 5 else 1 for i in range(len(ws))]
    b = Batch(ws, schemes=schemes)
    ref = [Lattice.from_workload(w, precision=32, scheme=s) for w, s in zip(ws, schemes)]

    def steps(n, skip=()):
        b.step(n)
        for i, lat in enumerate(ref):
            if i not in skip:
                for _ in range(n):
                    lat.step(1)
        for i, lat in enumerate(ref):
            assert np.array_equal(b.get_f(i), lat.get_f()), (n, i)

    launches = 0
    small = all(nx * ny <= 4096 for nx, ny in shapes)   # clusters, a launch per call
    for n in (1, 2, 3, 8, 53):
        steps(n)
        launches += 2 * (1 if small else n - max(0, (n - 1) // 2))   # a group for each scheme
        assert b.launch_count == launches
    b.residuals()
    for lat in ref:
        lat.diagnostics()
    steps(6)
    _, r = b.residuals()
    for i, lat in enumerate(ref):
        d = lat.diagnostics()[1][4]
        assert abs(r[i] - d) <= 1e-12 * d, i
    b.set_active(1, False)
    steps(5, skip=(1,))
    b.set_active(1, True)
    steps(7)
    b.close()
    c = Batch(ws + [_flow(63, 300, "walls")], schemes=schemes + [0])
    c.step(9)
    assert c.launch_count == 18
    c.close()
