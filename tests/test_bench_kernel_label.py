"""The benchmark names the kernel that ran: its lines are the library's, and a batch below a line is not called a pair."""
import os
import shutil
import subprocess

import pytest

import bench

HERE = os.path.dirname(os.path.abspath(__file__))


def test_lines_are_the_library_s(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "probe")
    subprocess.check_call([nvcc, "-std=c++17", "-O1", "-I" + os.path.join(os.path.dirname(HERE), "include"),
                           os.path.join(HERE, "launch_lines_probe.cpp"), "-o", exe])
    said = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert [int(x) for x in said] == [x for p in ("fp32", "int16", "int8") for x in bench.KERNEL_LINES[p]]


@pytest.mark.parametrize("kernel,batch,precision,name", [
    ("auto", 65536, "fp32", "msa_packed_kernel"), ("auto", 16384, "fp32", "msa_batch_kernel"),
    ("auto", 152 * 320, "fp32", "msa_batch_kernel"), ("auto", 152 * 320 + 1, "fp32", "msa_packed_kernel"),
    ("auto", 2048, "fp32", "msa_latency_kernel"), ("auto", 16384, "int16", "msa_packed_kernel"),
    ("auto", 6000, "int8", "msa_batch_kernel"), ("batch", 65536, "fp32", "msa_batch_kernel"),
    ("packed", 1000, "int8", "msa_packed_kernel")])
def test_label(kernel, batch, precision, name):
    assert bench.kernel_label(kernel, batch, 152, precision) == name
