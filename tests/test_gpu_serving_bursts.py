"""Bursts of equal requests to the server: which of them share the job table's
launches, and that a request gives the same bits alone and in any burst."""
import numpy as np
import pytest

import oracle
from paper_2004_09883_gb300 import inputs

pytestmark = pytest.mark.gpu
FWD, INV = -1, 1


def burst(fb, n, batch, count, direction=FWD, slots=1):
    """`count` requests handed over in one call; (results, inputs, kernel launches)."""
    import torch
    dims = list(n) if isinstance(n, tuple) else [n]
    vals = int(np.prod(dims)) * batch
    xs = [torch.from_numpy(inputs.normal_c64((vals,), 8100 + vals + i)).cuda() for i in range(count)]
    ys = [torch.zeros_like(x) for x in xs]
    torch.cuda.synchronize()
    with fb.Server(slots=slots, hbm_cap_bytes=1 << 30) as srv:
        srv.prepare(dims, batch)
        l0 = fb.launch_count()
        assert not any(srv.submit_many(srv.requests([(tuple(dims), x.data_ptr(), y.data_ptr(), i, direction, batch)
                                                     for i, (x, y) in enumerate(zip(xs, ys))])))
        srv.drain()
        torch.cuda.synchronize()
        launches = fb.launch_count() - l0
        assert all(d[1] == 0 for d in srv.poll())
    return ys, xs, launches


def check(fb, y, x, n, batch, direction=FWD):
    ref = oracle.fft(x.cpu().numpy().astype(np.complex128), [n], direction, False, 8)
    err = oracle.rel_l2(y.cpu().numpy().reshape(batch, n), ref.reshape(batch, n)).max()
    assert err <= 2e-6 * np.log2(n), (n, batch, err)


@pytest.mark.parametrize("n,batch", [(78125, 1), (78125, 8), (262440, 1), (500000, 1), (1 << 19, 1), (640000, 1)])
def test_requests_that_leave_the_gpu_idle_share_launches(fb, n, batch):
    """Below the size at which a request's own launches keep the GPU busy: one
    launch per phase for the whole burst, and the bits of a lone request."""
    import torch
    ys, xs, launches = burst(fb, n, batch, 6)
    assert launches == 2, launches
    alone, _, _ = burst(fb, n, batch, 1)
    assert torch.equal(alone[0], ys[0])
    check(fb, ys[5], xs[5], n, batch)


@pytest.mark.parametrize("n,batch", [(729000, 1), (500000, 2), (1 << 21, 1)])
def test_large_long_requests_run_their_plan(fb, n, batch):
    """From that size on each runs its plan's two passes, alone and in a burst."""
    import torch
    ys, xs, launches = burst(fb, n, batch, 3, INV)
    assert launches == 6, launches
    alone, _, one = burst(fb, n, batch, 1, INV)
    assert one == 2 and torch.equal(alone[0], ys[0])
    check(fb, ys[2], xs[2], n, batch, INV)


@pytest.mark.parametrize("dims,counts", [((512, 512), (1, 2, 3)), ((1 << 18,), (1, 2, 3)), ((100, 100), (1, 16)),
                                         ((16384,), (1, 37, 38)), ((64, 64, 64), (1, 2, 3)), ((45, 24, 50), (1, 7)),
                                         ((2048,), (1, 64)), ((60,), (1, 64)), ((157464,), (1, 2, 4)),
                                         ((3, 1000), (1, 20))])
@pytest.mark.parametrize("direction", [FWD, INV])
def test_narrow_and_wide_tiles_give_the_same_bits(fb, dims, counts, direction):
    """Launches of fewer tiles than the GPU has SMs run in narrower tiles: the same
    request alone, in bursts on both sides of that limit, and against the oracle."""
    import torch
    first = None
    for count in counts:
        ys, xs, _ = burst(fb, dims, 1, count, direction)
        first = ys[0] if first is None else first
        assert torch.equal(first, ys[0]), count
        n = int(np.prod(dims))
        ref = oracle.fft(xs[-1].cpu().numpy().astype(np.complex128), list(dims), direction, False, 8)
        err = oracle.rel_l2(ys[-1].cpu().numpy().reshape(1, n), ref.reshape(1, n)).max()
        assert err <= 2e-6 * np.log2(n), (dims, count, err)
