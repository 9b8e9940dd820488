"""The composite-radix line pass run on the host, butterfly by butterfly, from
the kernel's own headers: every 5-smooth length up to 4096, every layout, full
and ragged tiles, and the run-time shapes the batched-uneven kernel's jobs
take (up to 2048 points, radices up to 16).  No shared-memory slot outside its buffer, written twice or
read unwritten, every output written once, and each line equal to the DFT
within the FP32 bound of the shortest lengths (2e-6)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_composite_radix_pass_on_the_host(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "mr"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                    f"-I{ROOT}/include", f"-I{ROOT}/paper_2004_09883_gb300/csrc",
                    os.path.join(ROOT, "tests", "mr_host.cu"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out[0] == "mr_pass" and int(out[1]) > 1500
    assert int(out[2]) == 0
    assert float(out[3]) < 2e-6
    # four-step rows reading the columns' own tiles
    assert out[4] == "row_blocks" and int(out[5]) > 100 and int(out[6]) == 0
    assert out[8] == "uneven_jobs" and int(out[9]) > 1000
    assert int(out[10]) == 0
    assert float(out[11]) < 2e-6
