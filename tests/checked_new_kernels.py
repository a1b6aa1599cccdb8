"""Configurations that take the many-step, the two-step and the cluster kernels, for the
checked build (device bounds checks), and the runner that steps them with whichever library
the process loaded; see checked_cases.py.

Run as a script (``python tests/checked_new_kernels.py OUT.npz``) under LBM_CHECKED=1 it
builds and loads the checked library and raises on a failed bounds check."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))

from test_gpu_chain import _flow  # noqa: E402

STEPS = (1, 3, 20)

SINGLES = [(nx, ny, kind) for kind in ("periodic", "walls", "walls_mask", "periodic_mask", "side_walls")
           for nx, ny in ((3000, 67), (505, 401), (64, 3200), (256, 100), (101, 307), (540, 40), (5, 5000))]
BATCHES = {"chains": [(64, 65), (65, 16), (505, 40), (112, 200), (113, 33)],
           "clusters": [(3, 3), (64, 64), (17, 240), (300, 5), (5, 4), (512, 8)]}
KINDS = ("periodic", "walls", "walls_mask", "periodic_mask", "side_walls", "force")


def run_all():
    """{name: final populations}; the launch counts say that the kernels meant ran."""
    from paper_2103_02119_gb300 import lbm
    from paper_2103_02119_gb300.lbm import Batch, Lattice
    out = {}
    for nx, ny, kind in SINGLES:
        for scheme in (0, 1):
            g = Lattice.from_workload(_flow(nx, ny, kind), precision=32, scheme=scheme)
            for n in STEPS:
                g.step(n)
                st, _ = g.diagnostics()
                if st not in (lbm.LBM_OK, lbm.LBM_ERR_UNSTABLE):
                    raise RuntimeError(f"{nx} x {ny} {kind}: status {st}")
            if g.launch_count >= sum(STEPS):
                raise RuntimeError(f"{nx} x {ny} {kind}: a launch per step")
            out[f"{nx}x{ny}_{kind}_s{scheme}"] = g.get_f()
            g.close()
    for name, sizes in BATCHES.items():
        for scheme in (0, 1):
            ws = [_flow(nx, ny, KINDS[k % len(KINDS)]) for k, (nx, ny) in enumerate(sizes)]
            b = Batch(ws, schemes=[scheme] * len(ws))
            for n in STEPS:
                b.step(n)
                b.residuals()         # raises LbmError on a failed bounds check
            if b.launch_count >= sum(STEPS):
                raise RuntimeError(f"{name}: a launch per step")
            for k in range(len(ws)):
                out[f"{name}_s{scheme}_{k}"] = b.get_f(k)
            b.close()
    return out


if __name__ == "__main__":
    assert os.environ.get("LBM_CHECKED") == "1"
    from paper_2103_02119_gb300 import build
    build.build(checked=True)
    from paper_2103_02119_gb300 import lbm
    assert lbm.lib.lbm_build_flags() & lbm.LBM_BUILD_CHECKED
    res = run_all()
    np.savez(sys.argv[1], **res)
    print(f"checked build: {len(res)} final states, no bounds check failed")
