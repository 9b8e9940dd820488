"""The work that programs hand to this FFT block, as cases that can be timed and compared.

Six kinds of call stand for it, each through the public binding (``fbfft``):

* ``lines``   -- a batch of 1-D transforms of one length that fits one pass (64 ... 4096 points);
* ``long``    -- 1-D transforms above that (8192 ... 2^22 points, run as a four-step pair), with or
                 without the tensor-core option;
* ``grid``    -- 2-D fields, forward and then scaled inverse (a spectral solver's step);
* ``volume``  -- 3-D fields, the same;
* ``uneven``  -- one batch of 1-D transforms of many different lengths (``PlanMany``);
* ``served``  -- a burst of requests of mixed shapes handed to the request server at once.

Lengths are 2^a 3^b 5^c, as the planner takes them.  Plans, the server and its resident shapes are
made in :func:`prepare`, as a program does that transforms array after array with them.
"""
import math

import numpy as np
import torch

from paper_2004_09883_gb300 import fbfft, inputs, serving


def listed():
    return [
        # one small call (a spectrometer's frame): latency, launches and a short dependent chain count
        {"name": "lines_4096x64", "kind": "lines", "n": 4096, "batch": 64, "inverse": False},
        # a large batch of the longest power-of-two line that takes one pass: memory bound
        {"name": "lines_4096x16384", "kind": "lines", "n": 4096, "batch": 16384, "inverse": False},
        # decimal-sized frames, a ragged batch, the scaled inverse
        {"name": "lines_1000x20001", "kind": "lines", "n": 1000, "batch": 20001, "inverse": True},
        # the grid of the FFT application that the block replaces
        {"name": "grid_2048x2048", "kind": "grid", "dims": "2048,2048", "batch": 1},
        # a stack of odd-sided images: no row but the first starts on a 16-byte boundary
        {"name": "grid_375x405_b32", "kind": "grid", "dims": "375,405", "batch": 32},
        # a power-of-two simulation volume
        {"name": "volume_256x256x128", "kind": "volume", "dims": "256,256,128", "batch": 1},
        # a volume sized to its sample, not to a power of two
        {"name": "volume_120x150x144_b4", "kind": "volume", "dims": "120,150,144", "batch": 4},
        # long records, power of two
        {"name": "long_2p20x32", "kind": "long", "n": 1 << 20, "batch": 32, "inverse": False, "tensor_cores": False},
        # the same with the radix-16 stages on the tensor cores
        {"name": "long_2p20x32_tc", "kind": "long", "n": 1 << 20, "batch": 32, "inverse": False,
         "tensor_cores": True},
        # long records of a decimal length, scaled inverse
        {"name": "long_1000000x16", "kind": "long", "n": 1000000, "batch": 16, "inverse": True,
         "tensor_cores": False},
        # 4096 transforms of lengths log-uniform in [64, 65536] in one call
        {"name": "uneven_4096", "kind": "uneven", "count": 4096, "mix": 2004_09885},
        # 256 waiting requests (1-D up to 2^22, 2-D up to 512^2, 3-D up to 128^3) drained at once
        {"name": "served_256", "kind": "served", "count": 256, "mix": 2004_09887},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _smooth(rng, lo, hi):
    """A 2^a 3^b 5^c length near a log-uniform draw from [lo, hi]."""
    x = _log_uniform(rng, lo, hi)
    return min(inputs.smooth_lengths(lo, hi), key=lambda n: abs(math.log(n / x)))


def _splits(n):
    """Whether a long length has two factors of at most 4096 points (else the planner refuses it)."""
    return any(n % d == 0 and n // d <= 4096 for d in range(1, math.isqrt(n) + 1))


def draw(rng):
    kind = rng.choice(["lines", "lines", "long", "grid", "volume", "uneven", "served"])
    if kind == "lines":
        n = _smooth(rng, 64, 4096)
        return {"kind": kind, "n": n, "batch": max(1, round(_log_uniform(rng, 1 << 18, 1 << 25) / n)),
                "inverse": rng.random() < 0.5}
    if kind == "long":
        n = 1 << rng.randint(13, 22) if rng.random() < 0.4 else 7
        while n == 7 or not _splits(n):
            n = _smooth(rng, 8192, 1 << 22)
        tensor_cores = n & (n - 1) == 0 and rng.random() < 0.5
        return {"kind": kind, "n": n, "batch": max(1, int(_log_uniform(rng, 1 << 20, 1 << 25) / n)),
                "inverse": rng.random() < 0.5, "tensor_cores": tensor_cores}
    if kind in ("grid", "volume"):
        lo, hi, rank = (32, 2048, 2) if kind == "grid" else (16, 256, 3)
        dims = [_smooth(rng, lo, hi) for _ in range(rank)]
        n = math.prod(dims)
        return {"kind": kind, "dims": ",".join(map(str, dims)),
                "batch": max(1, int(_log_uniform(rng, 1 << 18, 1 << 24) / n))}
    if kind == "uneven":
        return {"kind": kind, "count": round(_log_uniform(rng, 256, 4096)), "mix": rng.randrange(1 << 30)}
    return {"kind": kind, "count": round(_log_uniform(rng, 16, 256)), "mix": rng.randrange(1 << 30)}


def _dims(case):
    return [int(v) for v in case["dims"].split(",")] if "dims" in case else [case["n"]]


def _lengths(case):
    return inputs.uneven_lengths(case["count"], 64, 65536, case["mix"])


def _shapes(case):
    return serving.request_mix(case["count"], case["mix"])


def _uniform(count, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.rand(count, 2, device="cuda", generator=g) * 2 - 1)


def _normal(count, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(count, 2, device="cuda", generator=g))


def _slots(sizes):
    """Where each request's array starts in a program's device pool (256-byte steps), and the pool's values."""
    steps = [(n + 31) // 32 * 32 for n in sizes]
    return [sum(steps[:i]) for i in range(len(steps))], sum(steps)


def _values(case, seed):
    """The call's input array: normal for fields and long records, uniform for the rest."""
    if case["kind"] == "uneven":
        return _uniform(fbfft.many_layout(_lengths(case))[1], seed)
    if case["kind"] == "served":
        return _uniform(_slots([math.prod(s) for s in _shapes(case)])[1], seed)
    count = math.prod(_dims(case)) * case["batch"]
    return (_uniform if case["kind"] == "lines" else _normal)(count, seed)


def prepare(case, seed):
    kind = case["kind"]
    x = _values(case, seed)
    state = {"kind": kind, "x": x}
    if kind == "served":
        shapes = _shapes(case)
        state["y"] = torch.zeros_like(x)  # every request's result, in one pool as the inputs
        srv = fbfft.Server(slots=8, hbm_cap_bytes=4 * 10**9)
        for s in sorted(set(shapes)):
            srv.prepare(s)
        state["server"] = srv
        state["requests"] = fbfft.Server.requests(
            [(s, x.data_ptr() + 8 * at, state["y"].data_ptr() + 8 * at, i, fbfft.FORWARD)
             for i, (s, at) in enumerate(zip(shapes, _slots([math.prod(s) for s in shapes])[0]))])
        torch.cuda.synchronize()  # the server runs on its own streams
        return state
    state["y"] = torch.zeros_like(x)
    if kind == "uneven":
        state["plan"] = fbfft.PlanMany(_lengths(case))
    elif kind in ("grid", "volume"):
        state["z"] = torch.zeros_like(x)
        state["plan"] = fbfft.Plan(_dims(case), case["batch"], scale_inv_n=True)
    else:
        state["plan"] = fbfft.Plan(_dims(case), case["batch"], scale_inv_n=case["inverse"],
                                   tensor_cores=case.get("tensor_cores", False))
        state["direction"] = fbfft.INVERSE if case["inverse"] else fbfft.FORWARD
    return state


def run(state):
    kind = state["kind"]
    if kind == "served":
        srv = state["server"]
        if any(srv.submit_many(state["requests"])):
            raise RuntimeError("a request was refused")
        srv.drain()
        if any(rec[1] for rec in srv.poll()):
            raise RuntimeError("a request failed")
        return state["y"]
    plan = state["plan"]
    if kind in ("grid", "volume"):
        y = plan.exec(state["x"], state["y"], fbfft.FORWARD)
        return [y, plan.exec(y, state["z"], fbfft.INVERSE)]
    return plan.exec(state["x"], state["y"], state.get("direction", fbfft.FORWARD))


def _flops(n):
    return 5.0 * n * math.log2(n) if n > 1 else 0.0


def work(case):
    kind = case["kind"]
    if kind == "uneven":
        lens = [int(n) for n in _lengths(case)]
        return {"bytes": 16 * sum(lens), "flops": sum(map(_flops, lens))}
    if kind == "served":
        sizes = [math.prod(s) for s in _shapes(case)]
        return {"bytes": 16 * sum(sizes), "flops": sum(map(_flops, sizes))}
    n, batch = math.prod(_dims(case)), case["batch"]
    if kind in ("grid", "volume"):  # the field in, its spectrum and the restored field out
        return {"bytes": 24 * n * batch, "flops": 2 * _flops(n) * batch}
    return {"bytes": 16 * n * batch, "flops": _flops(n) * batch}


def exact(case, seed):
    kind = case["kind"]
    x = _values(case, seed).to(torch.complex128)
    if kind == "uneven":
        lens = _lengths(case)
        offs = np.cumsum((lens + 1) // 2 * 2) - (lens + 1) // 2 * 2  # each transform at an even offset
        y = torch.zeros(x.numel(), dtype=torch.complex128, device="cuda")
        for n in np.unique(lens):
            at = torch.from_numpy(offs[lens == n]).cuda()[:, None] + torch.arange(int(n), device="cuda")
            y[at] = torch.fft.fft(x[at])
        return y
    if kind == "served":
        shapes = _shapes(case)
        sizes = [math.prod(s) for s in shapes]
        y = torch.zeros(x.numel(), dtype=torch.complex128, device="cuda")
        for s, n, at in zip(shapes, sizes, _slots(sizes)[0]):
            y[at:at + n] = torch.fft.fftn(x[at:at + n].view(s)).reshape(-1)
        return y
    dims = _dims(case)
    axes = tuple(range(1, len(dims) + 1))
    v = x.view(case["batch"], *dims)
    if kind in ("grid", "volume"):
        return [torch.fft.fftn(v, dim=axes).reshape(-1), x]
    f = torch.fft.ifftn if case["inverse"] else torch.fft.fftn
    return f(v, dim=axes).reshape(-1)
