"""Placement of the composite-radix kernels' exchange buffers (host): the search
gives what counting every candidate from scratch gives, at well under its cost
(a batched-uneven plan places every job it has)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_placement_equals_the_plain_search(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "place"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                    f"-I{ROOT}/include", f"-I{ROOT}/paper_2004_09883_gb300/csrc",
                    os.path.join(ROOT, "tests", "mr_place_host.cu"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) > 2000 and int(out[1]) == 0
    assert float(out[2]) < 0.7 * float(out[3])
