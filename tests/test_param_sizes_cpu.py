"""Kernel parameters stay small: a merged launch of the mixed kernel carries up to
64 pass descriptors, copied at every launch (24 KB; with the batched-uneven
kernel's fields among them it was 30, and 16 to 64 lengths took 4 % longer)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "fft_uneven.cuh"
int main()
{
    std::printf("%zu %zu %zu\n", sizeof(fbfft::MultiArgs), sizeof(fbfft::LineArgs), sizeof(fbfft::UnevenInlineArgs));
    return 0;
}
"""


def test_parameter_sizes(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "sizes.cu", tmp_path / "sizes"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", f"-I{ROOT}/include",
                    f"-I{ROOT}/paper_2004_09883_gb300/csrc", str(src), "-o", str(exe)], check=True)
    multi, line, inline = map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert multi <= 25 * 1024 and line <= 1024 and inline <= 8 * 1024
