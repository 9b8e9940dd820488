"""Large grids whose passes run on two kinds of kernel: starting each pass while the
one before drains must not cost time (FB_FFT_PDL=0 turns the early starts off)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import torch
from paper_2004_09883_gb300 import fbfft
x = torch.zeros(1 << 24, dtype=torch.complex64, device="cuda")
y = torch.zeros_like(x)
best = []
with fbfft.Plan([4096, 128], 32) as p:
    for _ in range(12):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(20):
            p.exec(x, y)
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b))
print(min(best))
"""


def test_mixed_passes_do_not_lose_by_overlap():
    def run(pdl):
        env = dict(os.environ, FB_FFT_PDL=pdl, PYTHONPATH=ROOT)
        return float(subprocess.run([sys.executable, "-c", PROGRAM], env=env, cwd=ROOT, capture_output=True, text=True,
                                    check=True).stdout.split()[-1])
    plain, overlapped = run("0"), run("1")
    assert overlapped <= 1.12 * plain, (overlapped, plain)
