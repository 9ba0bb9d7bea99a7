"""Kernels set up while their predecessor still runs: chains in which every call
reads what the one before wrote, over buffers written again each step, give the
bits they give when the host waits between the calls."""
import numpy as np
import pytest
import torch

from paper_1412_1127_gb300 import api

pytestmark = pytest.mark.gpu

STEPS = 6


class Chain:
    def __init__(self, length, mode, seed):
        g = torch.Generator().manual_seed(seed)
        self.n, self.mode = length, mode
        self.x = torch.randn(length, length, generator=g).cuda()
        self.c, self.y = torch.empty_like(self.x), torch.empty_like(self.x)
        total = length * length
        self.off = np.arange(0, total + 1, 7 if total % 7 == 0 else length, dtype=np.int64)
        f = lambda *s: torch.zeros(*s, device="cuda")
        self.rows, self.segs = f(STEPS, length), f(STEPS, len(self.off) - 1)
        self.whole, self.bat = f(STEPS, 2), f(STEPS, 2)
        self.d2, self.idx = f(STEPS, 5), torch.zeros(STEPS, 5, dtype=torch.int64, device="cuda")
        self.stats = torch.zeros(STEPS, 2, dtype=torch.float64, device="cuda")

    def run(self, stream, wait):
        k = max(1, min(5, self.n * self.n // 2))
        with torch.cuda.stream(stream):
            for i in range(STEPS):
                half = self.n // 2
                flat = self.y.view(-1)
                calls = [
                    lambda: api.accr_matmul_nest(self.x, self.x, self.c, mode=self.mode),
                    lambda: api.accr_standardize(self.c.view(-1), flat, self.stats[i]),
                    lambda: api.accr_rowreduce(self.y, [api.clause("add", self.rows[i])]),
                    lambda: api.accr_segmented_reduce(flat, self.off, [api.clause("max", self.segs[i])]),
                    lambda: api.accr_reduce(flat, [api.clause("add", self.whole[i, :1]),
                                                   api.clause("min", self.whole[i, 1:])]),
                    lambda: api.accr_reduce(self.whole[i], [api.clause("max", self.whole[i, 1:])]),
                    lambda: api.accr_batch_reduce([(self.rows[i, :half], [api.clause("add", self.bat[i, :1])], 0),
                                                   (self.rows[i, half:], [api.clause("add", self.bat[i, 1:])], 0)]),
                    lambda: api.accr_nearest_k(flat[:self.n * self.n // 2 * 2].view(-1, 2), 0.1, 0.2, k,
                                               self.idx[i], self.d2[i]),
                    lambda: api.accr_standardize(flat, self.x.view(-1), self.stats[i]),
                ]
                if i % 2:
                    calls.insert(2, lambda: self.y.mul_(1.5))  # another library's kernel in between
                for c in calls:
                    c()
                    if wait:
                        stream.synchronize()

    def results(self):
        return [t.clone() for t in (self.x, self.y, self.rows, self.segs, self.whole, self.bat, self.d2, self.idx,
                                    self.stats)]


@pytest.mark.parametrize("length,mode", [(1, "simt"), (3, "simt"), (64, "simt"), (65, "bf16x3"), (333, "simt"),
                                         (512, "bf16x3")])
def test_dependent_calls_without_waits(length, mode):
    want = Chain(length, mode, 1)
    want.run(torch.cuda.Stream(), wait=True)
    a, b = Chain(length, mode, 1), Chain(length, mode, 1)
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    a.run(sa, wait=False)  # two streams at once
    b.run(sb, wait=False)
    torch.cuda.synchronize()
    ref = want.results()
    for got in (a.results(), b.results()):
        for u, v in zip(ref, got):
            assert torch.equal(u.view(torch.uint8), v.view(torch.uint8))
