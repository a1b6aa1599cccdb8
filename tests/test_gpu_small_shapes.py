"""The small-lattice cluster kernel at the ends of its range: the widest rows a
CTA can hold (one row of 1365 cells), one column group, odd widths, bands of
one and of many rows; bit for bit the row-band kernel's states, and the
two buffers of the diagnostics' step-to-step change."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flow(nx, ny, kind):
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    if kind == "periodic":
        wl = W.taylor_green(nx, ny, 0.8, 0.19, 0.02, u0=0.02, seed=1).with_(Fx=1e-5, Fy=-2e-5)
    else:
        wl = W.cavity(nx, ny, 0.5, 0.075, 0.05, 100.0)
        m = np.zeros((ny, nx), np.uint8)
        m[ny // 2, nx // 3:nx // 2] = 1
        wl = wl.with_(mask=m, wall_u=((0.0, 0.01), (0.0, -0.02), (0.01, 0.0), (0.03, 0.0)))
    return wl.with_(rho=r, ux=u, uy=v)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("kind", ["periodic", "walls"])
@pytest.mark.parametrize("nx,ny", [(1365, 3), (3, 1365), (240, 17), (63, 65), (4, 4), (33, 31)])
def test_cluster_kernel_at_the_ends_of_its_range(nx, ny, kind, precision):
    from paper_2103_02119_gb300 import lbm
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, kind)
    for scheme in (0, 1):
        a = Lattice.from_workload(wl, precision=precision, scheme=scheme)
        b = Lattice.from_workload(wl, precision=precision, scheme=scheme)
        lbm.lbm_set_small_path(a.h, True)
        lbm.lbm_set_small_path(b.h, False)
        for n in (1, 2, 3, 20):
            a.step(n)
            b.step(n)
            assert np.array_equal(a.get_f(), b.get_f()), n
            assert np.array_equal(a.diagnostics()[1], b.diagnostics()[1]), n
        assert a.launch_count == 4 and b.launch_count == 26
        a.close()
        b.close()
