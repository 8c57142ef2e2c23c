"""Kernel attributes and SM counts belong to a device: the host code of the operator and coarse-solver
files, linked against a fake CUDA runtime with two devices of different sizes (tests/fake_devices.cpp),
must set a kernel's shared-memory limit on every device it launches on and size its work by the
device in use, whichever came first, from one thread or several."""
from fake_util import run_driver


def test_two_devices_in_one_process(tmp_path):
    run_driver("fake_devices.cpp", tmp_path)
