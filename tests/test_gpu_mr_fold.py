"""Strided composite-radix passes with short trailing extents: one tile takes the
lines of several outer indices.  Against the FP64 oracle (2e-6 * log2(N), as for
every FP32 pass), with guard bands, and that the tiles are filled."""
import math

import numpy as np
import pytest

import oracle
from paper_2004_09883_gb300 import inputs

pytestmark = pytest.mark.gpu
IN_PLACE = (480, 540, 1000)  # lengths whose CTA has an SM to itself


def strided_grid(fb, dims, batch):
    """CTAs of the first axis' pass (the last one launched)."""
    with fb.Plan(dims, batch) as p:
        return p.launch_config()[-1][0]


@pytest.mark.parametrize("n,lines", [(64, 16), (100, 16), (125, 16), (250, 16), (375, 8), (480, 8), (540, 8),
                                     (625, 4), (1000, 4), (1500, 4), (2000, 4)])
@pytest.mark.parametrize("cols", [2, 3, 4, 5, 6, 8, 9])
def test_short_trailing_extents(fb, n, lines, cols):
    """Lines of every tile width, trailing extents below, at and above half of it;
    batches that fill the last tile partly; 8-byte aligned arrays; in place."""
    import torch
    k = max(1, lines // cols)
    batch = (38 if n in IN_PLACE else 152) * k + k - 1  # the fewest outer indices that still fold k, and a ragged tile
    assert strided_grid(fb, [n, cols], batch) == (-(-batch // k) if k > 1 else batch * -(-cols // lines))
    total, lead, tail = n * cols * batch, 1, 3
    x = torch.view_as_complex(torch.randn(total, 2, device="cuda", generator=torch.Generator("cuda").manual_seed(n + cols)))
    pick = [0, 1, k, batch // 2, batch - 2, batch - 1]
    for direction, inplace in ((-1, False), (1, True)):
        buf = torch.full((lead + total + tail,), 7 + 3j, dtype=torch.complex64, device="cuda")
        out = buf[lead:lead + total]
        src = out if inplace else x
        out.copy_(x)
        with fb.Plan([n, cols], batch, scale_inv_n=True) as p:
            p.exec(src, out, direction)
            p.check()
        torch.cuda.synchronize()
        assert bool((buf[:lead] == 7 + 3j).all()) and bool((buf[lead + total:] == 7 + 3j).all())
        xs = x.view(batch, -1)[pick].cpu().numpy()
        ref = oracle.fft(xs.astype(np.complex128), [n, cols], direction, direction == 1, 8).reshape(len(pick), -1)
        err = oracle.rel_l2(out.view(batch, -1)[pick].cpu().numpy(), ref).max()
        assert err <= 2e-6 * math.log2(n * cols), (n, cols, direction, err)


@pytest.mark.parametrize("dims,batch", [([9, 250, 2], 100), ([3, 1000, 2], 211), ([128, 60, 4], 7)])
def test_middle_axes(fb, dims, batch):
    """The folded outer index runs over batch and leading axes."""
    import torch
    x = inputs.normal_c64((batch, int(np.prod(dims))), 5)
    d = torch.from_numpy(x).cuda()
    with fb.Plan(dims, batch) as p:
        y = p.exec(d.reshape(-1), None, -1).cpu().numpy().reshape(batch, -1)
    ref = oracle.fft(x.astype(np.complex128), dims, -1, False, 8).reshape(batch, -1)
    assert oracle.rel_l2(y, ref).max() <= 2e-6 * math.log2(np.prod(dims))


def test_few_outer_indices_keep_their_tiles(fb):
    """A single small field is not folded: its tiles would be too few."""
    assert strided_grid(fb, [250, 2], 303) == 303
    assert strided_grid(fb, [250, 2], 304) == 152
    assert strided_grid(fb, [540, 2], 75) == 75
    assert strided_grid(fb, [540, 2], 76) == 38
