"""A small region on one stream beside a queue of long calls on another: the long
calls' successors, set up early, do not keep it out."""
import time

import pytest
import torch

from paper_1412_1127_gb300 import api

pytestmark = pytest.mark.gpu


def long_calls(kind):
    f = lambda *s: torch.randn(*s, device="cuda")
    out = [torch.zeros(65536, device="cuda") for _ in range(2)]
    cl = [api.clause("add", out[0]), api.clause("max", out[1])]
    if kind == "region":
        x = f(1 << 28)
        return lambda s: api.accr_reduce(x, cl, stream=s)
    if kind == "rows":
        A = f(65536, 4096)
        return lambda s: api.accr_rowreduce(A, cl, stream=s)
    a = f(2048, 2048)
    c = torch.empty_like(a)
    return lambda s: api.accr_matmul_nest(a, a, c, mode="simt", stream=s)


@pytest.mark.parametrize("kind", ["region", "rows", "nest"])
def test_a_small_region_finds_room(kind):
    """These calls leave room for the small one while they run (the regions and rows
    half of an SM's threads, the nest a fifth of the SMs), so it waits for a part of one
    long call; shut out by a waiting successor it waits for one to the end and more."""
    call = long_calls(kind)
    x = torch.randint(-9, 9, (1 << 18,), dtype=torch.int32, device="cuda")
    o = torch.zeros(1, dtype=torch.int64, device="cuda")
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    small = lambda: api.accr_reduce(x, [api.clause("add", o)], stream=s2)
    event = lambda: torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    call(s1)
    small()
    torch.cuda.synchronize()
    a, b = event(), event()
    a.record(s1)
    for _ in range(10):
        call(s1)
    b.record(s1)
    torch.cuda.synchronize()
    one = a.elapsed_time(b) / 10
    waits = []
    for _ in range(8):
        ev = [(event(), event()) for _ in range(8)]
        torch.cuda.synchronize()
        for _ in range(14):
            call(s1)
        for e0, e1 in ev:
            time.sleep(0.0001)
            e0.record(s2)
            small()
            e1.record(s2)
        torch.cuda.synchronize()
        waits += [e0.elapsed_time(e1) for e0, e1 in ev]
    median = sorted(waits)[len(waits) // 2]
    assert median <= (0.5 if kind == "nest" else 1.2) * one, (median, one)
    assert int(o.item()) == int(x.sum().item())
