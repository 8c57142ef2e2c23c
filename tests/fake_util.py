"""Compiles a driver against the library's object files and a fake CUDA runtime (fake_cudart.h), and runs it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_03179_gb300", "csrc")
OBJECTS = ("sem_axl", "sem_ax8", "sem_ax8_x2", "sem_smooth8", "coarse_lat", "kernels")


def run_driver(source, tmp_path):
    from paper_2210_03179_gb300 import _build
    nvcc = shutil.which(_build._nvcc())
    if nvcc is None:
        pytest.skip("needs nvcc")
    _build.build()
    objs = [str(_build.BUILD / f"{n}.o") for n in OBJECTS]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    exe = str(tmp_path / "driver")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-w", f"-I{CSRC}", f"-I{include}", "-o", exe,
                        os.path.join(ROOT, "tests", source), *objs, "-fopenmp", "-pthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
