"""The composite-radix line pass on the GPU against the FP64 oracle: every
length with a factor 3 or 5 up to 4096 as contiguous lines (a ragged last tile,
a start on an odd 8-byte boundary), as strided lines, 3 and 25 of them
(ragged and odd tiles), and through four-step columns and rows of unequal
sizes.  Bar: 2e-6 * log2(N) per transform, as for every FP32 pass."""
import math

import numpy as np
import pytest

import oracle
from paper_2004_09883_gb300 import inputs

pytestmark = pytest.mark.gpu
LENGTHS = [n for n in inputs.smooth_lengths(2, 4096) if n & (n - 1)]


def run(fb, x, dims, batch, direction, lead=0, scale=False, inplace=False):
    """`lead` leading values shift the arrays off their 16-byte alignment."""
    import torch
    n = int(np.prod(dims)) * batch
    buf = torch.zeros(lead + n, dtype=torch.complex64, device="cuda")
    d = buf[lead:]
    d.copy_(torch.from_numpy(x.reshape(-1)))
    out = d if inplace else torch.zeros(lead + n, dtype=torch.complex64, device="cuda")[lead:]
    with fb.Plan(dims, batch, scale_inv_n=scale) as p:
        p.exec(d, out, direction)
        p.check()
    torch.cuda.synchronize()
    return out.cpu().numpy()


def check(y, x, dims, direction, scale=False):
    n = int(np.prod(dims))
    ref = oracle.fft(np.asarray(x, np.complex64).astype(np.complex128), dims, direction, scale, 8)
    err = oracle.rel_l2(y.reshape(-1, n), ref.reshape(-1, n)).max()
    assert err <= 2e-6 * math.log2(n), (dims, direction, err)


@pytest.mark.parametrize("n", LENGTHS)
def test_contiguous_lines(fb, n):
    x = inputs.uniform_c64((701 if n <= 64 else 11, n), n)
    check(run(fb, x, [n], len(x), -1, lead=1), x, [n], -1)
    check(run(fb, x, [n], len(x), 1, scale=True, inplace=True), x, [n], 1, True)


@pytest.mark.parametrize("n", LENGTHS)
def test_strided_lines(fb, n):
    for cols, direction in ((3, -1), (25, 1)):
        x = inputs.normal_c64((2, n, cols), n + cols)
        check(run(fb, x, [n, cols], 2, direction, lead=cols & 1, inplace=cols == 25), x, [n, cols], direction)


@pytest.mark.parametrize("n", [4374, 5000, 6075, 10125, 15000, 62208, 93750, 3 * 5 ** 7, 2 ** 3 * 3 ** 9, 2430000])
@pytest.mark.parametrize("direction", [-1, 1])
def test_fourstep(fb, n, direction):
    x = inputs.normal_c64((3, n), n)
    check(run(fb, x, [n], 3, direction, lead=1, scale=True), x, [n], direction, direction == 1)


@pytest.mark.parametrize("n", [64, 128, 256, 512, 1024, 2048, 4096])
def test_power_of_two_lines(fb, n):
    """Powers of two below every size limit of the choice of kernel, ragged tiles."""
    x = inputs.uniform_c64(((1 << 18) // n + 3, n), n)
    check(run(fb, x, [n], len(x), -1, lead=1), x, [n], -1)
    check(run(fb, x, [n], len(x), 1, scale=True, inplace=True), x, [n], 1, True)
    if n <= 128:
        for cols, direction in ((3, -1), (25, 1)):
            z = inputs.normal_c64((2, n, cols), n + cols)
            check(run(fb, z, [n, cols], 2, direction, lead=cols & 1, inplace=cols == 25), z, [n, cols], direction)


@pytest.mark.parametrize("n,mib", [(64, 96), (128, 48), (128, 192), (256, 24), (256, 96), (256, 192), (512, 384),
                                   (2048, 160), (4096, 6)])
def test_power_of_two_limits(fb, n, mib):
    """The largest batch on one side of a size limit (MiB read and written), the
    smallest on the other, and a host-array call whose chunks lie below it."""
    import torch
    for batch in ((mib << 16) // n, ((mib + 1) << 16) // n):
        x = inputs.uniform_c64((batch, n), n + batch)
        y = run(fb, x, [n], batch, -1).reshape(batch, n)
        i = np.r_[0:3, batch // 2, batch - 3:batch]
        check(y[i], x[i], [n], -1)
        hx = torch.empty(batch * n, dtype=torch.complex64, pin_memory=True)
        hy = torch.empty(batch * n, dtype=torch.complex64, pin_memory=True)
        hx.numpy()[:] = x.reshape(-1)
        with fb.Plan([n], batch) as p:
            p.exec_host(hx.numpy(), hy.numpy(), -1)
        assert np.array_equal(hy.numpy().reshape(batch, n), y)
