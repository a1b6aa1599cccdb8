"""The range of the global diagnostics: a fluid cell with a stored deviation of 32 or
more in magnitude counts as not finite, in both precisions, and stays out of the
sums; below it everything is summed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1.0])


def _lattice(nx, ny, precision, **kw):
    from paper_2103_02119_gb300.lbm import Lattice
    return Lattice(nx, ny, 0.5, 0.075, [1.0] * 9, rho0=0.0, precision=precision, **kw)


def _check(g, f):
    """All entry points against numpy's sums over the cells in range.  rho0 = 0 and
    populations that are multiples of 2^-10: each cell's rho and momentum are exact, so
    what differs is the rounding of a quotient and two products a cell and of the sums."""
    from paper_2103_02119_gb300 import lbm
    inside = (np.abs(f) < 32.0).all(0)
    rho = f.sum(0)
    jx, jy = np.tensordot(EX, f, 1), 0.5 * np.tensordot(EY, f, 1)
    e = 0.5 * (jx * jx + jy * jy) / rho
    bad = int((~inside).sum())
    for st, d in (g.diagnostics(), lbm.lbm_diagnostics_noalloc(g.h)):
        assert st == (lbm.LBM_ERR_UNSTABLE if bad else lbm.LBM_OK)
        assert d[5] == bad
        if bad:
            assert np.isnan(d[0])
        else:
            assert d[0] == rho.sum()
        for got, q in ((d[1], jx), (d[2], jy), (d[3], e)):
            q = q[inside]
            assert abs(got - q.sum()) <= (q.size + 8) * 2.0 ** -52 * np.abs(q).sum()


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("value", [1.75, 2.0, 31.0, 31.75, 32.0, 40.0, 63.0, 63.75, 64.0, 4096.0, -31.75, -32.0, -63.0, -64.0])
def test_one_population_at_the_limit(precision, value):
    g = _lattice(40, 12, precision)
    f = np.random.default_rng(3).integers(64, 256, (9, 12, 40)) / 1024.0
    f[0, 5, 7] = value
    f[:, 5, 8] *= 2
    g.set_f(f)
    _check(g, f)
    g.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_cells_on_both_sides_of_the_limit(precision):
    """What a flow that blows up holds: many cells of every size, an odd shape."""
    rng = np.random.default_rng(5)
    f = rng.integers(64, 256, (9, 301, 19)) / 1024.0
    hit = rng.random(f.shape) < 0.05
    f[hit] += np.round(rng.uniform(0.0, 90.0, int(hit.sum())) * 1024.0) / 1024.0
    assert ((np.abs(f) >= 32.0).any(0) & (np.abs(f) < 64.0).all(0)).sum() > 200
    g = _lattice(19, 301, precision)
    g.set_f(f)
    _check(g, f)
    g.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_a_flow_that_blows_up(precision):
    """Tall vortices at a small aspect ratio grow out of range within a few steps."""
    from paper_2103_02119_gb300 import workloads as W
    nx, ny, a = 18, 810, 0.5
    X, Y = np.meshgrid((np.arange(nx) + 0.5) * 2 * np.pi / nx, (np.arange(ny) + 0.5) * 2 * np.pi / ny)
    u0 = 0.02
    wl = W.taylor_green(nx, ny, a, 0.075, 0.02, u0=u0, seed=1).with_(
        rho=np.ones((ny, nx)), ux=u0 * np.sin(X) * np.cos(Y), uy=-u0 * ny * a / nx * np.cos(X) * np.sin(Y))
    g = _lattice(nx, ny, precision)
    g.init_fields(wl.rho, wl.ux, wl.uy)
    seen = 0
    for _ in range(6):
        g.step(1)
        f = g.get_f()
        size = np.abs(f).max(0)
        _, d = g.diagnostics()
        # (get_f returns the stored values: rho0 = 0)
        with np.errstate(all="ignore"):
            u = np.tensordot(EX, f, 1) / f.sum(0)
        assert d[5] == int((~(size < 32.0) | ~np.isfinite(u)).sum())
        seen += int(((size >= 32.0) & (size < 64.0)).sum())
    assert seen > 0
    g.close()
