"""Set-up and read-out kernels at the sizes where their launch shapes change.

Tolerances follow test_gpu_parity.test_fp32_setup_and_readout: FP32 values
within a few roundings of the deviations |f - w rho0| <~ 0.05.
"""
import numpy as np
import pytest

from paper_2103_02119_gb300 import workloads as W
from gpu_common import gpu_of, oracle_of

pytestmark = pytest.mark.gpu


def _flow(nx, ny, kind):
    wl = (W.taylor_green(nx, ny, 0.5, 0.075, 0.02, u0=0.02, seed=1) if kind == "periodic"
          else W.cavity(nx, ny, 0.5, 0.075, 0.04, 200.0))
    r, u, v = W.smooth_random_fields(nx, ny, 2, u_amp=0.02, rho_amp=2e-3)
    wl = wl.with_(rho=r, ux=u, uy=v)
    if kind == "mask":
        m = np.zeros((ny, nx), np.uint8)
        m[2:4, 2:nx // 2] = 1
        m[ny // 2:, nx // 3] = 1
        wl = wl.with_(mask=m)
    return wl


# bands of 1, 4 and 16 rows; segments of 256 columns with 255, 1 and 255 in the last
@pytest.mark.parametrize("nx,ny", [(255, 9), (257, 2433), (511, 9999)])
@pytest.mark.parametrize("kind", ["periodic", "walls", "mask"])
def test_fp32_setup_bands(orc, nx, ny, kind):
    wl = _flow(nx, ny, kind)
    o, g = oracle_of(orc, wl), gpu_of(wl, 32)
    assert float(np.abs(g.get_f() - o.get_f()).max()) <= 1e-7
    g.close()


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("nx,ny", [(31, 37), (33, 130), (65, 9), (129, 70), (300, 67)])
def test_readout_is_exact_over_the_range_of_the_storage(precision, nx, ny):
    """Distributions of all magnitudes (zeros, subnormals, values inside and
    outside the window in which the mass is summed as integers), on tiles of
    every width: stored as the nearest value of the storage type, read back
    unchanged, and their sum exact.  rho0 = 0, so that no rest part is added."""
    import math
    from paper_2103_02119_gb300.lbm import Lattice
    rng = np.random.default_rng(nx * ny + precision)
    f = rng.uniform(-1.9, 1.9, (9, ny, nx)) * 10.0 ** rng.integers(-36, 1, (9, ny, nx))
    f[:, : ny // 2] = rng.uniform(1e-9, 1.0, (9, ny // 2, nx))  # rows inside the window
    f[rng.random(f.shape) < 0.1] = 0.0
    f[3, 1, 2], f[5, 1, 2], f[0, 2, 2] = 1e-42, -3e-41, -0.0
    g = Lattice(nx, ny, 0.5, 0.075, [1.0] * 9, rho0=0.0, precision=precision)
    g.set_f(f)
    want = f.astype(np.float32).astype(np.float64) if precision == 32 else f
    got = g.get_f()
    assert np.array_equal(got, want)
    _, d = g.diagnostics()
    # 2^-144: the resolution of the mass, lost by the smallest values only
    assert abs(d[0] - math.fsum(want.ravel())) <= 9 * nx * ny * 2.0 ** -144 + 2.3e-16 * abs(d[0])
    g.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e30])
def test_readout_of_non_finite_and_large_values(value):
    from paper_2103_02119_gb300.lbm import LBM_ERR_UNSTABLE, Lattice
    g = Lattice(40, 12, 0.5, 0.075, [1.0] * 9, precision=32)
    f = g.get_f()
    f[0, 5, 7] = value
    g.set_f(f)
    got = g.get_f()
    assert np.array_equal(got[0, 5, 7], np.float64(np.float32(value)), equal_nan=True)
    f[0, 5, 7] = got[0, 5, 7] = 0.0
    assert float(np.abs(got - f).max()) <= 1e-8
    st, d = g.diagnostics()
    assert st == LBM_ERR_UNSTABLE and d[5] == 1
    g.close()
