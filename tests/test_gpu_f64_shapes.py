"""The automatic launch shape of middle-sized FP64 lattices: no slower than blocks of
their width with the automatic bands, just above multiples of 64 columns, where the
last segment is nearly empty."""
import pytest

from test_gpu_chain import _flow

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,block_x", [(65, 10616, 64), (65, 3385, 64), (129, 3101, 128), (193, 3576, 128), (300, 434, 128)])
def test_automatic_shape_is_no_slower(nx, ny, block_x):
    """At most 1.08 times (runs of one shape differ by a few percent)."""
    import torch
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, "periodic")
    times = []
    for bx in (0, block_x):
        g = Lattice.from_workload(wl, precision=64, block_x=bx, stream=torch.cuda.current_stream())
        g.step(10)
        best = 1e9
        for _ in range(8):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            g.step(20)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        times.append(best)
        g.close()
    assert times[0] <= 1.08 * times[1], times


@pytest.mark.parametrize("nx,ny,bands", [(619, 2512, 152), (2048, 879, 57), (2500, 461, 45), (619, 2262, 152)])
def test_no_short_second_wave(nx, ny, bands):
    """A few blocks more than one wave against bands that make one (three blocks of 128
    threads on each of 152 SMs): at most 1.08 times."""
    import torch
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, "periodic")
    times = []
    for kw in ({}, dict(block_x=128, bands=bands)):
        g = Lattice.from_workload(wl, precision=64, stream=torch.cuda.current_stream(), **kw)
        g.step(5)
        best = 1e9
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            g.step(10)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        times.append(best)
        g.close()
    assert times[0] <= 1.08 * times[1], times
