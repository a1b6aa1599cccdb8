"""The many-step kernel of middle-sized FP32 lattices: the states of single steps,
bit for bit, for the smallest number of rows a CTA can have, odd widths, uneven
bands, walls on each side, moving walls, both periodic wraps (the first and the last
CTA are neighbours), a force, both schemes and obstacles that touch every edge
and the rows between bands; the buffer one step earlier that the diagnostics read;
and a wait that runs out."""
import numpy as np
import pytest

from test_gpu_chain import _flow

pytestmark = pytest.mark.gpu

KINDS = ["periodic", "force", "side_walls", "walls", "walls_mask", "periodic_mask"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx,ny", [(256, 256), (101, 307), (1025, 4), (700, 7), (590, 8), (5, 1000), (63, 66), (37, 1999)])
def test_many_steps_match_single_steps(nx, ny, kind):
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, kind)
    for scheme in (0, 1):
        a = Lattice.from_workload(wl, precision=32, scheme=scheme)
        b = Lattice.from_workload(wl, precision=32, scheme=scheme)
        launches = 0
        for n in (13, 14, 17, 1, 2, 3, 60):
            a.step(n)
            for _ in range(n):
                b.step(1)
            # (short calls, and rows too wide for a CTA, take a launch per step)
            launches += n if n < (3 if nx * ny > 20480 else 14) or nx > 600 else 1
            assert np.array_equal(a.get_f(), b.get_f()), n
            # the step-to-step change and the residual read both buffers
            assert np.array_equal(a.diagnostics()[1], b.diagnostics()[1]), n
        assert a.launch_count == launches
        assert a.step_count == b.step_count == b.launch_count == 110
        a.close()
        b.close()


def test_longer_runs_take_several_launches():
    """More steps than one launch takes, then a rest too short for one."""
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(96, 90, "walls_mask")
    a = Lattice.from_workload(wl, precision=32)
    b = Lattice.from_workload(wl, precision=32)
    a.step(1024 + 3)
    for _ in range(79):
        b.step(13)
    assert a.launch_count == 1 + 3 and b.launch_count == 1027
    assert np.array_equal(a.get_f(), b.get_f())
    a.close()
    b.close()


def test_a_wait_that_runs_out_is_reported():
    """With no polls allowed the first wait for a neighbour ends the run: the next
    check reports it, and a fresh state steps as before."""
    from paper_2103_02119_gb300 import lbm as L
    wl = _flow(96, 90, "walls")
    a = L.Lattice.from_workload(wl, precision=32)
    L.lbm_set_wait_limit(a.h, 0)
    a.step(20)
    with pytest.raises(L.LbmError) as e:
        L.lbm_diagnostics(a.h)
    assert e.value.status == L.LBM_ERR_TIMEOUT
    L.lbm_set_wait_limit(a.h, 1 << 22)
    a.init_fields(wl.rho, wl.ux, wl.uy)
    b = L.Lattice.from_workload(wl, precision=32)
    a.step(20)
    for _ in range(20):
        b.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close()
    b.close()
