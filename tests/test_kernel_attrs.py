"""The opt-in to more than 48 KB of shared memory is made once for each device that a kernel runs on (tests/kernel_attrs_probe.cpp
runs the library's function against fakes of the CUDA calls: a sequence of launches on two devices)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_opt_in_per_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "probe")
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(os.path.dirname(HERE), "include"),
                           os.path.join(HERE, "kernel_attrs_probe.cpp"), "-o", exe])
    said = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]
    assert [x for x in said if x.startswith("rc")] == ["rc 0"] * 9
    assert [x for x in said if x.startswith("set")] == ["set 0 60000", "set 1 60000", "set 0 70000", "set 1 65000", "set 1 70000"]
