"""The copy-engine form of the composite-radix strided passes (tiles of 4 or 8 lines
moved by TMA into one buffer): every length that has it, and the odd ones that
work in one buffer without it, aligned, with trailing extents that are and are
not whole tiles, out of place and in place, inside guard bands; four-step pairs
with it on both sides; its bounded wait.  Bar against the FP64 oracle: 2e-6 *
log2(N)."""
import math
import time

import numpy as np
import pytest

import oracle
from paper_2004_09883_gb300 import inputs

pytestmark = pytest.mark.gpu
LENGTHS = [384, 405, 432, 480, 486, 540, 576, 600, 640, 648, 675, 720, 729, 750, 768, 800, 810, 864, 900, 960, 972,
           1000]
GUARD = 4096
MARK = 12345.5 - 9876.25j


def run(fb, x, dims, direction, inplace=False, lead=0):
    """The exec's values; arrays at a 16-byte boundary, or `lead` values past one."""
    import torch
    flat = torch.from_numpy(x.reshape(-1)).cuda()
    n = flat.numel()
    bufs = [torch.full((n + 2 * GUARD,), MARK, dtype=torch.complex64, device="cuda") for _ in range(2)]
    src, dst = (b[GUARD + lead:GUARD + lead + n] for b in bufs)
    src.copy_(flat)
    with fb.Plan(dims, len(x), scale_inv_n=True) as p:
        p.exec(src, src if inplace else dst, direction)
        p.check()
    torch.cuda.synchronize()
    out = src if inplace else dst
    for b in bufs:
        assert bool((b[:GUARD + lead] == MARK).all()) and bool((b[GUARD + lead + n:] == MARK).all())
    if not inplace:
        assert torch.equal(src, flat)
    return out.cpu().numpy().reshape(len(x), -1)


def check(y, x, dims, direction):
    n = int(np.prod(dims))
    ref = oracle.fft(x.astype(np.complex128), dims, direction, direction == 1, 8).reshape(len(x), n)
    err = oracle.rel_l2(y, ref).max()
    assert err <= 2e-6 * math.log2(n), (dims, direction, err)


def copied_by_tma(fb, dims, batch):
    """Whether the timeout switch (announced bytes that never arrive) reaches the plan's strided pass."""
    import torch
    x = torch.zeros(int(np.prod(dims)) * batch, dtype=torch.complex64, device="cuda")
    y = torch.zeros_like(x)
    with fb.Plan(dims, batch) as p:
        p.debug_inject_timeout(True)
        p.exec(x, y)
        try:
            p.check()
        except fb.FFTError as e:
            assert e.status == -5
            return True
        return False


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("cols", [10, 18, 64])
def test_strided_lines(fb, n, cols):
    x = inputs.normal_c64((3, n, cols), n + cols)
    fwd = run(fb, x, [n, cols], -1)
    check(fwd, x, [n, cols], -1)
    inv = run(fb, x, [n, cols], 1, inplace=True)
    check(inv, x, [n, cols], 1)
    plain = run(fb, x, [n, cols], -1, lead=1)  # 8-byte aligned: the plain-load form of the same kernel
    check(plain, x, [n, cols], -1)


@pytest.mark.parametrize("n1,n2", [(1000, 1000), (576, 1000), (384, 486), (640, 972), (405, 432)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_fourstep(fb, n1, n2, direction):
    """Both factors in the copy-engine form; with and without the columns' own tiles in between."""
    n = n1 * n2
    x = inputs.normal_c64((2, n), n)
    y = run(fb, x, [n], direction)
    check(y, x, [n], direction)
    check(run(fb, x, [n], direction, lead=1), x, [n], direction)


def test_wait_runs_out_once(fb):
    """Copies that never arrive: the exec ends after about one wait however many
    waves of tiles it has, reports the time-out, and the plan works afterwards."""
    import torch
    dims, batch = [1000, 64], 60  # 960 tiles, one CTA per SM
    x = inputs.normal_c64((batch, 64000), 3)
    d = torch.from_numpy(x).cuda().reshape(-1)
    y = torch.zeros_like(d)
    with fb.Plan(dims, batch) as p:
        p.exec(d, y)
        torch.cuda.synchronize()
        p.debug_inject_timeout(True)
        t0 = time.perf_counter()
        p.exec(d, y)
        with pytest.raises(fb.FFTError) as e:
            p.check()
        assert e.value.status == -5
        assert time.perf_counter() - t0 < 3.0
        p.debug_inject_timeout(False)
        p.exec(d, y)
        p.check()
    check(y.cpu().numpy().reshape(batch, -1)[:2], x[:2], dims, -1)


def test_the_form_is_reached(fb):
    for dims in ([384, 10], [486, 18], [1000, 64]):
        assert copied_by_tma(fb, dims, 1), dims
    # lengths without the one-buffer form, and odd ones (no box of whole 128-byte rows): plain loads
    for dims in ([250, 64], [405, 18]):
        assert not copied_by_tma(fb, dims, 1), dims
