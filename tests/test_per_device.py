"""Kernel attributes and SM counts belong to a device: the host code of the operator and coarse-solver
files, linked against a fake CUDA runtime with two devices of different sizes (tests/fake_devices.cpp),
must set a kernel's shared-memory limit on every device it launches on and size its work by the
device in use, whichever came first, from one thread or several."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_03179_gb300", "csrc")


def test_two_devices_in_one_process(tmp_path):
    from paper_2210_03179_gb300 import _build
    nvcc = _build._nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip("needs nvcc")
    _build.build()
    names = ("sem_axl", "sem_ax8", "sem_ax8_x2", "sem_smooth8", "coarse_lat", "kernels")
    objs = [str(_build.BUILD / f"{n}.o") for n in names]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    exe = str(tmp_path / "fake_devices")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(nvcc)))), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-w", f"-I{CSRC}", f"-I{include}", "-o", exe,
                        os.path.join(ROOT, "tests", "fake_devices.cpp"), *objs, "-fopenmp", "-pthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
