"""The small-lattice cluster kernel at the ends of its range: the widest rows a
CTA can hold (one row of 1365 cells), one column group, odd widths, bands of
one and of many rows; bit for bit the row-band kernel's states, and the
two buffers of the diagnostics' step-to-step change."""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flow(nx, ny, kind):
    r, u, v = W.smooth_random_fields(nx, ny, 5, u_amp=0.02, rho_amp=2e-3)
    if kind == "periodic":
        wl = W.taylor_green(nx, ny, 0.8, 0.19, 0.02, u0=0.02, seed=1).with_(Fx=1e-5, Fy=-2e-5)
    else:
        wl = W.cavity(nx, ny, 0.5, 0.075, 0.05, 100.0)
        m = np.zeros((ny, nx), np.uint8)
        m[ny // 2, nx // 3:nx // 2] = 1
        wl = wl.with_(mask=m, wall_u=((0.0, 0.01), (0.0, -0.02), (0.01, 0.0), (0.03, 0.0)))
    return wl.with_(rho=r, ux=u, uy=v)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("kind", ["periodic", "walls"])
@pytest.mark.parametrize("nx,ny", [(1365, 3), (3, 1365), (240, 17), (63, 65), (4, 4), (33, 31)])
def test_cluster_kernel_at_the_ends_of_its_range(nx, ny, kind, precision):
    from paper_2103_02119_gb300 import lbm
    from paper_2103_02119_gb300.lbm import Lattice
    wl = _flow(nx, ny, kind)
    for scheme in (0, 1):
        a = Lattice.from_workload(wl, precision=precision, scheme=scheme)
        b = Lattice.from_workload(wl, precision=precision, scheme=scheme)
        lbm.lbm_set_small_path(a.h, True)
        lbm.lbm_set_small_path(b.h, False)
        for n in (1, 2, 3, 20):
            a.step(n)
            b.step(n)
            assert np.array_equal(a.get_f(), b.get_f()), n
            assert np.array_equal(a.diagnostics()[1], b.diagnostics()[1]), n
        assert a.launch_count == 4 and b.launch_count == 26
        a.close()
        b.close()


def _batch_flows(sizes):
    return [_flow(nx, ny, "periodic" if k % 2 else "walls") for k, (nx, ny) in enumerate(sizes)]


# one CTA a lattice and several; more CTAs than rows; rows wider than a CTA's
# threads; a lattice above 4096 cells (the whole batch then takes the band
# kernel: one launch a step)
@pytest.mark.parametrize("sizes,launches", [
    ([(16, 16)], 4), ([(64, 64), (3, 3), (17, 240), (33, 31)], 4), ([(300, 5), (40, 7)], 4),
    ([(20, 24)] * 160, 4), ([(1365, 3), (16, 16)], 4), ([(65, 64), (16, 16)], 1131)])
def test_batches_of_small_lattices(sizes, launches):
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    ws = _batch_flows(sizes)
    b = Batch(ws)
    pick = sorted(set([0, 1, 2, len(ws) - 1]) & set(range(len(ws))))
    ref = {k: Lattice.from_workload(
        ws[k] if ws[k].mask is not None else ws[k].with_(mask=np.zeros((ws[k].ny, ws[k].nx), np.uint8)),
        precision=32) for k in pick}
    for n in (1, 30, 1100):                 # 1100 steps: two launches of a cluster kernel
        b.step(n)
        for k in pick:
            ref[k].step(n)
            # (a flow that blows up does so alike)
            assert np.array_equal(b.get_f(k), ref[k].get_f(), equal_nan=True), (k, n)
    assert b.launch_count == launches
    if len(ws) > 1:                         # one leaves for an odd number of steps
        b.set_active(0, False)
        b.step(7)
        b.set_active(0, True)
        b.step(4)
        ref[0].step(4)
        for k in pick[1:]:
            ref[k].step(11)
        for k in pick:
            assert np.array_equal(b.get_f(k), ref[k].get_f(), equal_nan=True), k
    b.close()
