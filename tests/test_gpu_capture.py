"""Calls of 50 steps and more on a stream that is being captured: a replay of the caller's
graph takes the steps that the call would have taken."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STILL = ((0.0, 0.0),) * 4


def _flow(nx, ny, px):
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    return W.cavity(nx, ny, 0.5, 0.075, 0.05, 400.0).with_(rho=r, ux=u, uy=v, periodic_x=px, wall_u=STILL)


def _captured(torch, stream, step):
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    graph.replay()
    torch.cuda.synchronize()


# the row-band kernel's runs before the two-step kernel, that kernel alone, the many-step
# kernel, the two-step kernel, the clusters; FP64
@pytest.mark.parametrize("nx,ny,px,precision", [
    (900, 90, 0, 32), (64, 6000, 0, 32), (50, 4000, 0, 32), (256, 256, 0, 32), (500, 500, 1, 32),
    (40, 40, 0, 32), (300, 200, 0, 64)])
@pytest.mark.parametrize("steps", [60, 102])
def test_captured_steps(nx, ny, px, precision, steps):
    import torch
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, px)
    stream = torch.cuda.Stream()
    a = Lattice.from_workload(wl, precision=precision, stream=stream)
    b = Lattice.from_workload(wl, precision=precision)
    a.step(1)
    _captured(torch, stream, lambda: a.step(steps))
    b.step(1 + steps)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny,count", [(640, 6, 8), (24, 24, 8), (64, 200, 4), (30, 200, 4)])
def test_captured_batch_steps(nx, ny, count):
    import torch
    from paper_2103_02119_gb300.lbm import Batch
    wls = [_flow(nx, ny, k % 2) for k in range(count)]
    stream = torch.cuda.Stream()
    a = Batch(wls, stream=stream)
    a.step(1)
    _captured(torch, stream, lambda: a.step(60))
    b = Batch(wls)                    # (its tables replace a's on the device: after the replay)
    b.step(61)
    for k in range(count):
        assert np.array_equal(a.get_f(k), b.get_f(k)), k
    a.close()
    b.close()
