"""Calls of one step on small lattices: no slower than the kernels that take a launch a
step, and the same states."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _wl(nx, ny, seed):
    r, u, v = W.smooth_random_fields(nx, ny, seed, u_amp=0.02, rho_amp=2e-3)
    return W.cavity(nx, ny, 0.5, 0.075, 0.05, 100.0).with_(rho=r, ux=u, uy=v, mask=np.zeros((ny, nx), np.uint8))


def _time(step, reps=10):
    import torch
    best = 1e9
    for _ in range(8):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        for _ in range(reps):
            step()
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


def test_single_steps_of_many_small_lattices():
    """300 lattices of 64 x 64 in short bands, calls of one step, against the same and
    one lattice too large for the clusters (a launch a step for all): at most 1.3
    times."""
    import torch
    from paper_2103_02119_gb300.lbm import Batch
    ws = [_wl(64, 64, k) for k in range(300)]
    times = []
    for more in ([], [_wl(64, 65, 7)]):
        b = Batch(ws + more, stream=torch.cuda.current_stream())
        b.set_shape(32, 4)
        b.step(1)
        times.append(_time(lambda: b.step(1)))
        b.close()
    assert times[0] <= 1.3 * times[1], times


@pytest.mark.parametrize("rows", [4, 16])
def test_states_do_not_depend_on_the_calls(rows):
    """Single steps (row bands, or clusters where the bands are long), pairs and longer
    calls of a batch give the states of single-lattice steps."""
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    ws = [_wl(nx, ny, k) for k, (nx, ny) in enumerate([(64, 64), (33, 31), (5, 200), (300, 7)])]
    b = Batch(ws)
    b.set_shape(32, rows)
    ref = [Lattice.from_workload(w, precision=32) for w in ws]
    for n in (1, 1, 2, 1, 3, 7, 1):
        b.step(n)
        for k, lat in enumerate(ref):
            lat.step(n)
            assert np.array_equal(b.get_f(k), lat.get_f()), (n, k)
    for lat in ref:
        lat.close()
    b.close()
