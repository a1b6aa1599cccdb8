"""The checked build on the many-step, the two-step and the cluster kernels: no bounds
check fails, and the states are the normal build's bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

import checked_new_kernels as C

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_no_bounds_check_fails(tmp_path):
    out = tmp_path / "checked.npz"
    r = subprocess.run([sys.executable, os.path.join(HERE, "checked_new_kernels.py"), str(out)],
                       env=dict(os.environ, LBM_CHECKED="1"), capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-4000:]
    assert "no bounds check failed" in r.stdout
    got, ref = np.load(out), C.run_all()
    assert sorted(got.files) == sorted(ref)
    for k in ref:
        assert np.array_equal(got[k], ref[k], equal_nan=True), k
