"""Large power-of-two passes on the persistent kernel (a whole number of CTAs per SM)
where it is the faster: strided lines of 128 points above 192 MiB, contiguous ones of
512 above 384; below, and with few columns, on the composite-radix one (a CTA per
tile)."""
import numpy as np
import pytest

import oracle
from paper_2004_09883_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,batch,which,persistent", [
    ([128, 512], 193, 1, True), ([128, 512], 192, 1, False), ([128, 32], 4096, 1, False), ([128, 64], 2048, 1, True),
    ([64, 512], 512, 1, False), ([512], 49280, 0, True), ([512], 49152, 0, False)])
def test_kernel_by_size(fb, dims, batch, which, persistent):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with fb.Plan(dims, batch) as p:
        grid = p.launch_config()[which][0]
    assert (grid % sms == 0 and grid <= 16 * sms) == persistent, grid


def test_strided_128_points_on_both_kernels(fb):
    """128 x 64 fields on both sides of the size limit, ragged tiles behind it, against the oracle."""
    import torch
    for dims, batch, direction in (([128, 64], 1536, -1), ([128, 64], 1544, -1), ([128, 100], 1100, 1)):
        n = int(np.prod(dims))
        x = inputs.normal_c64((batch, n), 11)
        d = torch.from_numpy(x).cuda().reshape(-1)
        with fb.Plan(dims, batch, scale_inv_n=True) as p:
            y = p.exec(d, None, direction).cpu().numpy().reshape(batch, n)
            p.check()
        pick = [0, batch // 2, batch - 1]
        ref = oracle.fft(x[pick].astype(np.complex128), dims, direction, direction == 1, 8).reshape(len(pick), n)
        assert oracle.rel_l2(y[pick], ref).max() <= 2e-6 * np.log2(n)
