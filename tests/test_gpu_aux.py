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
