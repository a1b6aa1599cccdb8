"""Lattices of 64 columns between walls at rest: which kernel steps them (by the
number of launches), and the states."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STILL = ((0.0, 0.0),) * 4


def _wl(nx, ny, kind):
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    wl = W.cavity(nx, ny, 0.5, 0.075, 0.05, 400.0).with_(rho=r, ux=u, uy=v, wall_u=STILL,
                                                         periodic_x=int(kind == "channel"))
    if kind == "lid":
        wl = wl.with_(wall_u=STILL[:3] + ((0.03, 0.0),))
    if kind == "mask":
        wl = wl.with_(mask=W.random_obstacles(nx, ny, seed=3, coverage=0.05))
    return wl


@pytest.mark.parametrize("nx,ny,kind,two", [
    (64, 6000, "walls", False), (64, 6000, "mask", False), (64, 6000, "lid", True), (64, 6000, "channel", True),
    (64, 5000, "walls", True), (65, 6000, "walls", True), (66, 6000, "mask", True)])
def test_route_of_single_lattices(nx, ny, kind, two):
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _wl(nx, ny, kind)
    a, b = (Lattice.from_workload(wl, precision=32) for _ in range(2))
    a.step(9)
    assert a.launch_count == (5 if two else 9)
    for _ in range(9):
        b.step(1)
    assert np.array_equal(a.get_f(), b.get_f())
    a.close()
    b.close()


@pytest.mark.parametrize("sizes,kind,rows,launches", [
    ([(64, 300)] * 4, "walls", 4, 9), ([(64, 65)], "walls", 1, 9), ([(64, 300)] * 4, "walls", 16, 5),
    ([(64, 300)] * 4, "lid", 4, 5), ([(64, 300)] * 4, "channel", 4, 5), ([(66, 300)] * 4, "walls", 4, 5),
    ([(64, 300), (64, 300), (200, 300)], "walls", 4, 5)])
def test_route_of_batches(sizes, kind, rows, launches):
    """Short bands: a launch a step where most cells are in such lattices."""
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    ws = [_wl(nx, ny, kind).with_(mask=np.zeros((ny, nx), np.uint8)) for nx, ny in sizes]
    b = Batch(ws)
    b.set_shape(32, rows)
    b.step(9)
    assert b.launch_count == launches
    for k, w in enumerate(ws):
        lat = Lattice.from_workload(w, precision=32)
        lat.step(9)
        assert np.array_equal(b.get_f(k), lat.get_f())
        lat.close()
    b.set_shape(32, 16)                       # long bands: two steps a launch
    b.step(9)
    assert b.launch_count == launches + 5
    b.close()
