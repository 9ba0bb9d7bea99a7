"""Stretches little longer than their full rounds of vectors: the partial round's forms
(one vector a thread, half a round, more) at their edges, and that a few vectors more do
not cost a whole round."""
import numpy as np
import pytest
import torch

from paper_1412_1127_gb300 import api

pytestmark = pytest.mark.gpu

TD = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32, "f64": torch.float64}


def whole_numbers(shape, t, seed):
    g = np.random.default_rng(seed)
    return torch.from_numpy(g.integers(-2000, 2000, shape)).to(TD[t]).cuda()


@pytest.mark.parametrize("t", ["i32", "i64", "f32", "f64"])
@pytest.mark.parametrize("vectors", [257, 287, 288, 289, 383, 384, 385, 511, 513, 545, 640, 641])
def test_rows_and_segments(t, vectors):
    """Whole numbers, so every sum is exact; rounds of 256 vectors a warp."""
    epv = 4 if t in ("i32", "f32") else 2
    for cols in (vectors * epv - 1, vectors * epv, vectors * epv + epv - 1):
        for pad in (0, 1):
            A = whole_numbers((21, cols + pad), t, cols)[:, :cols]
            s, m, x = (torch.zeros(21, dtype=TD[t], device="cuda") for _ in range(3))
            api.accr_rowreduce(A, [api.clause("add", s), api.clause("max", m)])
            api.accr_rowreduce(A, [api.clause("min", x)])
            assert torch.equal(s, A.sum(1).to(TD[t])) and torch.equal(m, A.amax(1)) and torch.equal(x, A.amin(1))
        flat = whole_numbers(21 * cols + 1, t, cols)
        off = np.arange(22, dtype=np.int64) * cols + 1
        S = flat[1:].view(21, cols)
        for cl, want in (([("add", s)], [S.sum(1)]), ([("min", m), ("add", s), ("max", x)], [S.amin(1), S.sum(1), S.amax(1)])):
            api.accr_segmented_reduce(flat, off, [api.clause(op, o) for op, o in cl])
            for (_, o), w in zip(cl, want):
                assert torch.equal(o, w.to(TD[t]))


@pytest.mark.parametrize("t", ["i32", "f64"])
@pytest.mark.parametrize("vectors", [1, 255, 256, 257, 1024, 1025, 2047, 2048, 2049, 4095])
def test_batch_regions_and_tiles(t, vectors):
    epv = 4 if t == "i32" else 2
    acc = torch.int64 if t == "i32" else torch.float64
    old = api.accr_batch_tiling(small_bytes=4096)  # longer ones by CTAs, 2,048 vectors a round
    try:
        xs = [whole_numbers(vectors * epv + d, t, d) for d in range(epv)]
        out = torch.zeros(len(xs), dtype=acc, device="cuda")
        api.accr_batch_reduce([(x, [api.clause("add", out[i:i + 1])], 0) for i, x in enumerate(xs)])
        assert out.tolist() == [x.sum().item() for x in xs]
    finally:
        api.accr_batch_tiling(*old)


def micros(fn, n=20):
    for _ in range(3):
        fn()
    best = float("inf")
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


def test_a_few_vectors_more_cost_little():
    """Rows of 262 vectors of doubles against rows of 375: fewer bytes and fewer folds."""
    t = []
    for cols in (525, 750):
        A = torch.randn(50000, cols, dtype=torch.float64, device="cuda")
        s = torch.zeros(50000, dtype=torch.float64, device="cuda")
        t.append(micros(lambda: api.accr_rowreduce(A, [api.clause("add", s)])))
    assert t[0] <= 1.1 * t[1], t
