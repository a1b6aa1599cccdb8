"""Checkpoints: the raw bytes of a state do not depend on how its steps were split
into calls, the row padding among them (odd widths with a force, where the
padding takes what the collision makes of an empty cell)."""
import pytest

from test_gpu_chain import _flow

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["periodic", "force", "walls", "walls_mask", "periodic_mask"])
@pytest.mark.parametrize("nx,ny", [(61, 53), (255, 257), (101, 307), (33, 300), (37, 1999), (505, 401), (64, 70)])
def test_raw_state_bytes_do_not_depend_on_the_calls(nx, ny, kind):
    from paper_2103_02119_gb300 import lbm
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, kind).with_(Fx=1e-5, Fy=-2e-5)
    for scheme in (0, 1):
        a = Lattice.from_workload(wl, precision=32, scheme=scheme)
        b = Lattice.from_workload(wl, precision=32, scheme=scheme)
        if nx * ny <= 4096:                    # the same kernel family for both
            lbm.lbm_set_small_path(a.h, False)
            lbm.lbm_set_small_path(b.h, False)
        for n in (20, 3, 31, 60):
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert a.get_state() == b.get_state(), n
        a.close()
        b.close()
