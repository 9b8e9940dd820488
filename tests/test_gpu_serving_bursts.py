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
