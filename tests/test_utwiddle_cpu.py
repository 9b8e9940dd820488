"""Twiddles the batched-uneven kernel forms from the powers it reads, on the host.

Bound: a table entry is off by at most sqrt(2) 2^-25 (each component rounded), an
FP32 complex product adds at most sqrt(5) 2^-24 to the errors of its factors; the
longest chain is w^4m times (w times w times w): four entries' and three products'
errors (w^2 = w w, w^3 = w^2 w, then times w^4m), and one more product with a value
of 1."""
import math
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_formed_twiddles(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "utw"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                    f"-I{ROOT}/include", f"-I{ROOT}/paper_2004_09883_gb300/csrc",
                    os.path.join(ROOT, "tests", "utwiddle_host.cu"), "-o", str(exe)], check=True)
    bound = 4 * math.sqrt(2) * 2.0 ** -25 + 4 * math.sqrt(5) * 2.0 ** -24
    out = subprocess.run([str(exe), repr(bound)], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) > 50000 and int(out[1]) == 0, out
