"""The many-step kernel's launch on several devices, on the CPU with a fake CUDA
runtime: shared memory is allowed on every device that a lattice is made on, and
a device that does not take the launch gets none (its lattices step as others
do)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2103_02119_gb300", "csrc")


def test_shared_memory_is_allowed_on_each_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    obj, exe = str(tmp_path / "band_run.o"), str(tmp_path / "harness")
    include = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    flags = ["-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", *include]
    for cmd in ([nvcc, *flags, "-c", os.path.join(CSRC, "band_run.cu"), "-o", obj],
                [nvcc, *flags, "-cudart", "none",
                 os.path.join(HERE, "fake_cuda", "band_run_harness.cu"),
                 os.path.join(HERE, "fake_cuda", "runtime.cpp"), obj, "-o", exe]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "ok, 9 launches" in r.stdout, r.stdout + r.stderr
