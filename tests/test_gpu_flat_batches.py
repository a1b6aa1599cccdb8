"""Batches of wide, flat small lattices take the row-band kernel; a few among narrow
ones stay with the clusters.  The states are those of single-lattice steps."""
import numpy as np
import pytest

from test_gpu_short_calls import _wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,launches", [
    ([(1365, 3)], 50), ([(1024, 4)] * 4, 50), ([(700, 3), (513, 7), (16, 16)], 50),
    ([(512, 8)] * 4, 1), ([(512, 4), (200, 5)], 1), ([(1365, 3), (16, 16)], 1), ([(5, 3), (3, 4)], 1)])
def test_route_and_states(sizes, launches):
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    ws = [_wl(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    b = Batch(ws)
    b.step(50)
    assert b.launch_count == launches
    b.step(7)
    for k in range(min(3, len(ws))):
        lat = Lattice.from_workload(ws[k], precision=32)
        lat.step(57)
        assert np.array_equal(b.get_f(k), lat.get_f()), k
        lat.close()
    b.close()
