"""Set-up and read-out of very narrow and very flat lattices: the values, and that a
narrow lattice costs about what its cells cost."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, precision, mask=None):
    import torch

    from paper_2103_02119_gb300.lbm import Lattice
    return Lattice(nx, ny, 0.5, 0.075, [1.0] * 9, rho0=0.0, precision=precision, mask=mask,
                   stream=torch.cuda.current_stream())


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("nx,ny", [(3, 3), (3, 1001), (4, 77), (5, 300), (7, 333), (31, 9), (257, 5), (1000, 3), (2049, 4)])
def test_values(nx, ny, precision, masked):
    """Distributions of exact binary fractions: stored, read back, summed (mass and
    momenta, in the diagnostics and from the moments) as numpy does."""
    rng = np.random.default_rng(nx * ny)
    m = None
    if masked:
        m = np.zeros((ny, nx), np.uint8)
        m[ny // 2, nx // 2] = 1
    f = rng.integers(64, 256, (9, ny, nx)) / 1024.0
    if masked:
        f[:, m != 0] = 0.0
    g = _lattice(nx, ny, precision, m)
    g.set_f(f)
    assert np.array_equal(g.get_f(), f)
    ex, ey = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1]), 0.5 * np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    rho, jx, jy = f.sum(0), np.tensordot(ex, f, 1), np.tensordot(ey, f, 1)
    _, d = g.diagnostics()
    assert d[0] == math.fsum(f.ravel()) and d[1] == jx.sum() and d[2] == jy.sum() and d[5] == 0
    r, u, v = g.moments()
    fluid = np.ones((ny, nx), bool) if m is None else m == 0
    ulp = 2.0 ** (-22 if precision == 32 else -51)
    assert np.array_equal(r, rho)
    for got, j in ((u, jx), (v, jy)):
        want = np.where(fluid, j / np.where(fluid, rho, 1.0), 0.0)
        assert (np.abs(got - want) <= 2 * ulp * np.abs(want)).all()
    g.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_a_narrow_lattice_costs_what_its_cells_cost(precision):
    """3 x 100000 cells against 1000 x 300: at most four times the time (a row of three
    cells is read in 32-byte sectors, of which it uses 12 or 24 bytes, and the launch
    costs both the same)."""
    import torch

    from paper_2103_02119_gb300 import lbm
    times = {}
    for nx, ny in ((1000, 300), (3, 100000)):
        g = _lattice(nx, ny, precision)
        f = torch.full((9, ny, nx), 0.125, dtype=torch.float64, device="cuda")
        g.set_f(f)
        calls = {"get_f": lambda: lbm.lbm_get_f(g.h, g.N, f), "set_f": lambda: g.set_f(f),
                 "diagnostics": g.diagnostics}
        for name, call in calls.items():
            best = 1e9
            for _ in range(6):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                torch.cuda.synchronize()
                e[0].record()
                for _ in range(20):
                    call()
                e[1].record()
                torch.cuda.synchronize()
                best = min(best, e[0].elapsed_time(e[1]))
            times.setdefault(name, []).append(best)
        g.close()
    for name, (wide, narrow) in times.items():
        assert narrow <= 4.0 * wide, (name, times)


@pytest.mark.parametrize("masked", [False, True])
def test_setting_up_a_narrow_lattice(masked):
    """lbm_init_fields of 3 x 100000 FP32 cells against 1000 x 300: at most six times the
    time (as for the read-out, and a cell reads its nine neighbours' fields)."""
    import torch
    times = []
    for nx, ny in ((1000, 300), (3, 100000)):
        m = np.zeros((ny, nx), np.uint8) if masked else None
        if masked:
            m[ny // 2, nx // 2] = 1
        g = _lattice(nx, ny, 32, m)
        q = [torch.full((ny, nx), v, dtype=torch.float64, device="cuda") for v in (1.0, 0.01, -0.02)]
        best = 1e9
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(20):
                g.init_fields(*q)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        times.append(best)
        g.close()
    assert times[1] <= 6.0 * times[0], times


@pytest.mark.parametrize("kind", ["periodic", "force", "side_walls", "walls", "walls_mask", "periodic_mask"])
@pytest.mark.parametrize("nx,ny", [(3, 2432), (48, 2432), (48, 2431), (49, 2432), (17, 5001)])
def test_setup_at_the_edges_of_the_narrow_form(orc, nx, ny, kind):
    """Both forms of the FP32 set-up around the line between them, against the oracle's
    equilibria (within a few FP32 roundings of the deviations, as in
    test_gpu_parity.test_fp32_setup_and_readout)."""
    from gpu_common import gpu_of, oracle_of
    from test_gpu_chain import _flow
    wl = _flow(nx, ny, kind)
    o, g = oracle_of(orc, wl), gpu_of(wl, 32)
    assert float(np.abs(g.get_f() - o.get_f()).max()) <= 1e-7
    g.close()
