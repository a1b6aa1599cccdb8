"""The batch autotuner on small lattices: what it times has to depend on the shape."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(20, 24), (33, 31)], [(64, 65), (100, 40)]])
def test_every_trial_is_single_steps(sizes):
    """21 shapes, a warm-up step and the trial steps each: a launch for every one of
    them (clusters and the two-step kernel take none of the shapes), and the
    lattices go through the states of as many single-lattice steps."""
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    ws = []
    for k, (nx, ny) in enumerate(sizes):
        r, u, v = W.smooth_random_fields(nx, ny, k, u_amp=0.02, rho_amp=2e-3)
        ws.append(W.cavity(nx, ny, 0.5, 0.075, 0.05, 100.0).with_(
            rho=r, ux=u, uy=v, mask=np.zeros((ny, nx), np.uint8)))
    b = Batch(ws)
    ref = [Lattice.from_workload(w, precision=32) for w in ws]
    trial = 4
    b.tune(trial)
    assert b.launch_count == 21 * (trial + 1)
    b.step(9)                                  # the usual kernels again
    assert b.launch_count < 21 * (trial + 1) + 9
    for k, lat in enumerate(ref):
        lat.step(21 * (trial + 1) + 9)
        assert b.step_count(k) == lat.step_count
        assert np.array_equal(b.get_f(k), lat.get_f())
        lat.close()
    b.close()
