"""accr_segmented_reduce with segments above the warp limit: their tiles are folded in
the call's one launch, ahead of the others."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from paper_1412_1127_gb300 import api, inputs
from tolerances import same_bits

pytestmark = pytest.mark.gpu

TD = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32, "f64": torch.float64}
ND = {"i32": np.int32, "i64": np.int64, "f32": np.float32, "f64": np.float64}


@pytest.fixture
def small_tiles():
    """Warp segments up to 4 KiB and tiles of 8 KiB: tens of tiles in small arrays."""
    old = api.accr_batch_tiling(small_bytes=4096, tile_bytes=8192)
    yield 8192
    api.accr_batch_tiling(*old)


def lengths(eb, tile, seed):
    te = tile // eb
    edges = [k * te + d for k in (1, 2, 3, 7, 40) for d in (-1, 0, 1)] + [4096 // eb + 1, 300 * te + 5]
    g = np.random.default_rng(seed)
    L = np.concatenate([edges, g.integers(0, 60, 200), g.integers(te // 2, 6 * te, 60), [0, 0]])
    g.shuffle(L)
    return L.astype(np.int64)


@pytest.mark.parametrize("t", ["i32", "i64", "f32", "f64"])
@pytest.mark.parametrize("first", [0, 3])
def test_several_tiles_a_segment(t, first, small_tiles):
    eb = 4 if t in ("i32", "f32") else 8
    L = lengths(eb, small_tiles, first)
    off = inputs.offsets_from_lengths(L) + first
    n = int(off[-1])
    v = inputs.normal(n, ND[t], salt=first) if t[0] == "f" else inputs.full_range_i32(n, salt=first).astype(ND[t])
    vt = torch.from_numpy(v).cuda()
    acc = "i64" if t == "i32" else t
    ops = [("add", acc), ("max", t), ("min", t), ("mul" if t[0] == "f" else "bxor", t)]
    for nc in (1, 2, 3, 4):
        for rep in range(2):  # the counters are zero again
            outs = [guarded((len(L),), TD[a], 5) for _, a in ops[:nc]]
            before = api.accr_launch_count()
            api.accr_segmented_reduce(vt, off, [api.clause(op, o.t) for (op, _), o in zip(ops, outs)])
            assert api.accr_launch_count() - before == 1
            got = [o.check(op).cpu().numpy() for (op, _), o in zip(ops, outs)]
            for (op, a), x in list(zip(ops, got))[:3]:
                if op != "add" or t[0] != "f":
                    assert same_bits(x, oracle.segmented_reduce(v, off, op, a)), (nc, op)
            if nc == 4 and t[0] != "f":
                assert same_bits(got[3], oracle.segmented_reduce(v, off, "bxor", t))
            if t[0] == "f":
                u = 2.0 ** -24 if t == "f32" else 2.0 ** -53
                for k in range(len(L)):
                    seg = v[off[k]:off[k + 1]].astype(np.float64)
                    assert abs(float(got[0][k]) - seg.sum()) <= (len(seg) + 2) * (u + 2.0 ** -53) * np.abs(seg).sum(), k
                if rep:
                    assert same_bits(got[0], again)
                again = got[0]


@pytest.mark.parametrize("t", ["i32", "f32", "f64"])
def test_tiles_of_the_default_size(t):
    """One tile, exactly one, one and an element, several; alone and among short ones."""
    eb = 4 if t != "f64" else 8
    te = api.ACCR_TILE_BYTES // eb
    for L in ([65536 // eb + 1], [te, te + 1, 3 * te - 1], [5, 0, 2 * te, 17, 65536 // eb, 70000 // eb, 3, te - 1, 900]):
        off = inputs.offsets_from_lengths(np.array(L, dtype=np.int64)) + 1
        v = inputs.normal(int(off[-1]), ND[t]) if t[0] == "f" else inputs.full_range_i32(int(off[-1]))
        s, m = guarded((len(L),), TD["i64" if t == "i32" else t], 5), guarded((len(L),), TD[t], 5)
        api.accr_segmented_reduce(torch.from_numpy(v).cuda(), off, [api.clause("max", m.t), api.clause("add", s.t)])
        assert same_bits(m.check("max").cpu().numpy(), oracle.segmented_reduce(v, off, "max", t))
        got = s.check("sum").cpu().numpy()
        if t == "i32":
            assert np.array_equal(got, oracle.segmented_reduce(v, off, "add", "i64"))
        else:
            for k in range(len(L)):
                seg = v[off[k]:off[k + 1]].astype(np.float64)
                assert abs(float(got[k]) - seg.sum()) <= 1e-5 * np.abs(seg).sum() + 0.0


def test_a_batch_in_between():
    """A call's tile counters and a batch's share words that every kernel returns to zero."""
    te = api.ACCR_TILE_BYTES // 4
    off = np.array([0, 3 * te + 7, 5 * te, 5 * te + 9], dtype=np.int64)
    v = inputs.full_range_i32(int(off[-1]))
    vt = torch.from_numpy(v).cuda()
    want = oracle.segmented_reduce(v, off, "add", "i64")
    b = torch.zeros(40, dtype=torch.int64, device="cuda")
    for _ in range(3):
        s = torch.zeros(3, dtype=torch.int64, device="cuda")
        api.accr_segmented_reduce(vt, off, [api.clause("add", s)])
        api.accr_batch_reduce([(vt[i * 1000:i * 1000 + (3 * te if i % 3 == 0 else 50)], [api.clause("add", b[i:i + 1])], 0)
                               for i in range(40)])
        assert np.array_equal(s.cpu().numpy(), want)
    for i in range(40):
        assert b[i].item() == int(v[i * 1000:i * 1000 + (3 * te if i % 3 == 0 else 50)].astype(np.int64).sum())


def micros(fn, n=30):
    for _ in range(5):
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


def test_a_second_clause_costs_little():
    """A sum and a maximum of segments with some long ones, against the sum alone."""
    g = np.random.default_rng(5)
    off = np.concatenate([[0], np.cumsum(np.exp(g.uniform(0, np.log(31853), 1060)).astype(np.int64))])
    v = torch.randn(int(off[-1]), device="cuda")
    s, m = torch.zeros(1060, device="cuda"), torch.zeros(1060, device="cuda")
    one = micros(lambda: api.accr_segmented_reduce(v, off, [api.clause("add", s)]))
    two = micros(lambda: api.accr_segmented_reduce(v, off, [api.clause("add", s), api.clause("max", m)]))
    assert two <= 1.25 * one, (two, one)
