"""Middle-sized FP32 lattices with wide rows: where the many-step kernel starts and ends
(by the number of launches), and the states on both sides."""
import numpy as np
import pytest

from test_gpu_chain import _flow

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,kind,steps,launches", [
    (400, 100, "walls", 3, 1), (401, 100, "walls", 4, 4), (401, 100, "walls", 5, 1), (401, 100, "walls_mask", 4, 4),
    (440, 180, "periodic", 4, 4), (440, 304, "periodic", 4, 3), (440, 306, "periodic", 3, 1), (437, 67, "periodic", 4, 4),
    (560, 60, "periodic", 60, 1), (561, 60, "periodic", 9, 9), (561, 60, "periodic_mask", 9, 1),
    (596, 200, "force", 9, 5), (596, 202, "force", 9, 1), (590, 8, "periodic", 14, 1)])
def test_route_and_states(nx, ny, kind, steps, launches):
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, kind)
    a, b = (Lattice.from_workload(wl, precision=32) for _ in range(2))
    a.step(steps)
    assert a.launch_count == launches
    for _ in range(steps):
        b.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    assert np.array_equal(a.diagnostics()[1], b.diagnostics()[1])
    a.close()
    b.close()
