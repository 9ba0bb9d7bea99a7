"""A row's or segment's sum has the same bits whatever other clauses stand beside it:
kernels with fixed codes and the generic ones add in the same order."""
import numpy as np
import pytest
import torch

from paper_1412_1127_gb300 import api

pytestmark = pytest.mark.gpu

TD = {"f32": torch.float32, "f64": torch.float64}
BESIDE = [[], ["max"], ["min"], ["max", "min"], ["mul"]]


def values(n, t, seed):
    g = np.random.default_rng(seed)
    x = g.standard_normal(n) * np.exp2(g.integers(-8, 9, n))
    return torch.from_numpy(x.astype(np.float32 if t == "f32" else np.float64)).cuda()


def sums(call, n, t, flags):
    out = []
    for ops in BESIDE:
        for first in (True, False):
            s = torch.zeros(n, dtype=TD[t], device="cuda")
            rest = [api.clause(op, torch.zeros(n, dtype=TD[t], device="cuda")) for op in ops]
            call([api.clause("add", s)] + rest if first else rest + [api.clause("add", s)], flags)
            out.append(((ops, first), s))
    torch.cuda.synchronize()
    return out


def check(out, what):
    ref = out[0][1].view(torch.uint8)
    bad = [k for k, s in out if not torch.equal(s.view(torch.uint8), ref)]
    assert not bad, (what, bad)


@pytest.mark.parametrize("t,flags", [("f32", 0), ("f32", api.ACCR_COMPENSATED), ("f64", 0)])
@pytest.mark.parametrize("cols", [1, 3, 5, 7, 13, 17, 31, 61, 64, 100, 129, 255, 257, 300, 511, 513, 800, 1000, 1023, 1500,
                                  5000, 20001, 70003])
@pytest.mark.parametrize("pad,off", [(0, 0), (3, 1), (2, 3)])
def test_rows(t, flags, cols, pad, off):
    rows = 37
    A = values(rows * (cols + pad + off), t, cols).view(rows, -1)[:, off:off + cols]
    check(sums(lambda cl, fl: api.accr_rowreduce(A, cl, flags=fl), rows, t, flags), cols)


@pytest.mark.parametrize("t,flags", [("f32", 0), ("f32", api.ACCR_COMPENSATED), ("f64", 0)])
@pytest.mark.parametrize("first", [0, 1, 3])
def test_segments(t, flags, first):
    g = np.random.default_rng(first)
    L = np.concatenate([g.integers(0, 40, 400), np.exp(g.uniform(0, np.log(3000), 300)).astype(np.int64),
                        g.integers(1000, 40000, 12)])
    g.shuffle(L)
    off = np.concatenate([[0], np.cumsum(L)]).astype(np.int64) + first
    x = values(int(off[-1]), t, 9)
    check(sums(lambda cl, fl: api.accr_segmented_reduce(x, off, cl, flags=fl), len(L), t, flags), "segments")


@pytest.mark.parametrize("t", ["f64", "i64"])
@pytest.mark.parametrize("cols", [1, 2, 3, 7, 8, 9, 13, 16, 33, 61, 64, 65, 128, 255, 256, 257, 300, 511, 512, 513, 600])
@pytest.mark.parametrize("pad,off", [(0, 0), (1, 1)])
def test_short_rows_of_eight_bytes(t, cols, pad, off):
    """Every lane count and both widths of the row groups, with an odd base and pad."""
    rows = 45
    g = np.random.default_rng(cols)
    big = g.integers(-(1 << 40), 1 << 40, (rows, cols + pad + off))
    if t == "f64":
        big = big / (1 << 20)
    A = torch.from_numpy(big).cuda()[:, off:off + cols]
    M = big[:, off:off + cols]
    d = torch.float64 if t == "f64" else torch.int64
    s, a, m = (torch.zeros(rows, dtype=d, device="cuda") for _ in range(3))
    api.accr_rowreduce(A, [api.clause("add", s)])
    api.accr_rowreduce(A, [api.clause("min", m), api.clause("add", a)])
    assert np.array_equal(m.cpu().numpy(), M.min(1))
    if t == "i64":
        assert np.array_equal(s.cpu().numpy(), M.sum(1)) and np.array_equal(a.cpu().numpy(), M.sum(1))
    else:  # a rounding of 2^-53 of the sum of magnitudes for each value at most
        for got in (s, a):
            assert np.all(np.abs(got.cpu().numpy() - M.sum(1)) <= 2 * cols * 2.0 ** -53 * np.abs(M).sum(1))
