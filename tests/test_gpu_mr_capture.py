"""The first exec of a fresh composite-radix plan inside a stream capture: its
kernels are loaded and checked when the plan is made."""
import numpy as np
import pytest

import oracle
from paper_2004_09883_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,batch", [([2916], 5), ([972, 50], 2), ([1080 * 1215], 1)])
def test_first_exec_under_capture(fb, dims, batch):
    import torch
    n = int(np.prod(dims))
    x = inputs.normal_c64((batch, n), n)
    d = torch.from_numpy(x).cuda().reshape(-1)
    y, z = torch.zeros_like(d), torch.zeros_like(d)
    with fb.Plan(dims, batch, scale_inv_n=True) as p:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.exec(d, y, -1)
            p.exec(y, z, 1)
        g.replay()
        torch.cuda.synchronize()
        p.check()
    ref = oracle.fft(x.astype(np.complex128), dims, -1, False, 8).reshape(batch, n)
    assert oracle.rel_l2(y.cpu().numpy().reshape(batch, n), ref).max() <= 2e-6 * np.log2(n)
    assert oracle.rel_l2(z.cpu().numpy().reshape(batch, n), x.astype(np.complex128)).max() <= 4e-6 * np.log2(n)
