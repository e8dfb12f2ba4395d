"""Registers of the learned decoders on long rows: a row's messages and its weights are not all held at once.  What ptxas
reports for rows up to 32 may spill no more than the kernels did that read each weight by itself where it is used (bytes of
spill stores below) and one group: 16 bytes of weights and 8 of their address.  (A spill is a trip to local memory in
every check of every iteration.)"""
import os
import re
import shutil
import subprocess

import pytest

from paper_2508_07879_gb300 import build

GROUP = 16 + 8
KERNELS = [   # kernel, template arguments after the precision, bytes of spill stores with a weight at a time
    ("msa_batch_kernel", "32, false, 4, true", 0),
    ("msa_batch_kernel", "32, false, 8, true", 72),
    ("msa_latency_kernel", "32, false, 4, 2, true", 4),
    ("msa_latency_kernel", "32, false, 16, 2, true", 324),
    ("msa_server_kernel", "32, false, 8, true", 52),
]


def test_learned_long_rows_spill_no_more(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    jobs = []
    for i, (name, args, _) in enumerate(KERNELS):
        server = name == "msa_server_kernel"
        src = tmp_path / f"k{i}.cu"
        src.write_text('#include "%s"\ntemplate __global__ void qldpc::kern::%s<qldpc::kern::F32, %s>(const %sqldpc::%s);\n'
                       % ("server_kernel.cuh" if server else "msa_kernel.cuh", name, args,
                          "__grid_constant__ " if name == "msa_batch_kernel" else "", "ServerParams" if server else "LaunchParams"))
        jobs.append(subprocess.Popen([nvcc, *build.ARCH, *build.NVCC_FLAGS, "-I" + build.CSRC, "-I" + build.INCLUDE, "-c", str(src),
                                      "-o", str(tmp_path / f"k{i}.o")], stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True))
    for (name, args, most), job in zip(KERNELS, jobs):
        said = job.communicate()[0]
        assert job.returncode == 0, said
        spills = [int(x) for x in re.findall(r"(\d+) bytes spill stores", said)]
        assert len(spills) == 1 and spills[0] <= most + GROUP, (name, args, spills, most)
