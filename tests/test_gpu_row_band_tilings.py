"""The row-band kernel's tilings in both precisions, a launch per step: FP32 calls of
several steps take the many-step or the two-step kernel at these sizes, which the block
width and the bands do not shape."""
import pytest

from gpu_common import compare, gpu_of, pair
from test_gpu_parity import _fields
from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("nx,ny,masked", [(300, 70, False), (301, 71, True), (515, 260, False)])
def test_narrow_tiles_match_the_oracle_and_wide_ones(orc, precision, periodic, nx, ny, masked):
    """64-column segments and 7-row bands against the oracle and, bit for bit, one
    512-column segment over the whole height, stepped one at a time; then
    against calls of several steps."""
    wl = _fields(W.cavity(nx, ny, 0.5, 0.075, 0.04, 150.0), 13)
    if periodic:
        wl = wl.with_(periodic_x=1, periodic_y=1, wall_u=((0.0, 0.0),) * 4)
    if masked:
        wl = wl.with_(mask=W.random_obstacles(nx, ny, seed=4, coverage=0.08))
    o, g = pair(orc, wl, precision, noise_seed=14, noise_amp=5e-4, block_x=32, bands=10)
    ref = gpu_of(wl, precision, block_x=256, bands=1)
    many = gpu_of(wl, precision)
    start = g.get_state()
    ref.set_state(start)
    many.set_state(start)
    o.step(9)
    for _ in range(9):
        g.step(1)
        ref.step(1)
    many.step(9)
    assert g.launch_count == ref.launch_count == 9
    compare(o, g, precision)
    assert ref.get_state() == g.get_state() == many.get_state()
