"""accr_segmented_reduce at the lengths where its forms meet: lane groups of 2, 8
and 32 (at most 4 KiB), a warp per segment (at most 64 KiB), tiles."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from paper_1412_1127_gb300 import _native, api, inputs
from tolerances import same_bits

pytestmark = pytest.mark.gpu

TD = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32, "f64": torch.float64}


def lengths(eb, seed):
    """Every edge of a form, a vector or an element more or less, among random short ones."""
    g = np.random.default_rng(seed)
    edges = [e // eb + d for e in (16, 256, 1024, 4096, 8192, 16384, 32768, 65536, 131072) for d in (-3, -1, 0, 1, 2)]
    L = np.concatenate([np.array([max(0, e) for e in edges]), g.integers(0, 40, 700), np.zeros(40, dtype=np.int64),
                        np.exp(g.uniform(0, np.log(1500), 500)).astype(np.int64)])
    g.shuffle(L)
    return L.astype(np.int64)


@pytest.mark.parametrize("t", ["i32", "i64", "f32", "f64"])
@pytest.mark.parametrize("first", [0, 1, 7])
def test_lengths_around_every_form(t, first):
    eb = 4 if t in ("i32", "f32") else 8
    L = lengths(eb, first)
    off = inputs.offsets_from_lengths(L) + first      # segments need not start at the array's start
    n = int(off[-1])
    nd = {"i32": np.int32, "i64": np.int64, "f32": np.float32, "f64": np.float64}[t]
    v = inputs.normal(n, nd, salt=first) if t[0] == "f" else inputs.full_range_i32(n, salt=first).astype(nd)
    vt = torch.from_numpy(v).cuda()
    acc = t if t != "i32" else "i64"
    s, m, x = guarded((len(L),), TD[acc], 5), guarded((len(L),), TD[t], 5), guarded((len(L),), TD[acc], 5)
    op3 = "mul" if t[0] == "f" else "bxor"
    api.accr_segmented_reduce(vt, off, [api.clause("add", s.t), api.clause("max", m.t)])
    api.accr_segmented_reduce(vt, off, [api.clause("min" if t[0] == "f" else op3, x.t, init=3)])
    s_np, m_np = s.check("sum").cpu().numpy(), m.check("max").cpu().numpy()
    assert same_bits(m_np, oracle.segmented_reduce(v, off, "max", t))
    assert same_bits(x.check("third").cpu().numpy(),
                     oracle.segmented_reduce(v, off, "min" if t[0] == "f" else op3, acc, init=3))
    if t[0] != "f":
        assert np.array_equal(s_np, oracle.segmented_reduce(v, off, "add", acc))
        return
    u = 2.0 ** -24 if t == "f32" else 2.0 ** -53
    for k in range(len(L)):
        seg = v[off[k]:off[k + 1]].astype(np.float64)
        assert abs(float(s_np[k]) - seg.sum()) <= (len(seg) + 2) * (u + 2.0 ** -53) * np.abs(seg).sum(), k


@pytest.mark.parametrize("nseg", [1, 15, 16, 17, 513])
def test_counts_and_empty_segments(nseg):
    v = inputs.full_range_i32(nseg * 3, salt=nseg)
    vt = torch.from_numpy(v).cuda()
    off = np.arange(nseg + 1, dtype=np.int64) * 3
    off[1:nseg // 2 + 1] = 0                            # the first half empty
    # a pair no kernel has fixed, its sum second
    p, a = guarded((nseg,), torch.int64, 5), guarded((nseg,), torch.int64, 5)
    api.accr_segmented_reduce(vt, off, [api.clause("mul", p.t, init=7), api.clause("add", a.t, init=-2)])
    assert np.array_equal(p.check("product").cpu().numpy(), oracle.segmented_reduce(v, off, "mul", "i64", init=7))
    assert np.array_equal(a.check("sum").cpu().numpy(), oracle.segmented_reduce(v, off, "add", "i64", init=-2))


def test_decreasing_offsets_are_refused_anywhere():
    v = torch.zeros(100000, dtype=torch.int32, device="cuda")
    out = torch.full((3000,), 9, dtype=torch.int64, device="cuda")
    for at in (1, 511, 512, 513, 2999):
        off = np.arange(3001, dtype=np.int64) * 20
        off[at] = off[at + 1 if at < 3000 else at] + 1
        with pytest.raises(_native.AccrError) as e:
            api.accr_segmented_reduce(v, off, [api.clause("add", out)])
        assert e.value.code == _native.ACCR_EINVAL
    with pytest.raises(_native.AccrError):
        api.accr_segmented_reduce(v, np.array([-1, 5]), [api.clause("add", out)])
    assert bool((out == 9).all())


@pytest.mark.slow
def test_offsets_past_32_bits():
    n = (1 << 32) + 4096
    v = torch.zeros(n, dtype=torch.int32, device="cuda")
    v[-4000:] = torch.arange(4000, dtype=torch.int32, device="cuda")
    off = np.array([0, n - 4000, n - 3990, n - 3000, n - 2999, n - 5, n - 5, n], dtype=np.int64)
    out = guarded((7,), torch.int64, 5)
    api.accr_segmented_reduce(v, off, [api.clause("add", out.t)])
    want = [int(np.arange(a, b).sum()) for a, b in [(0, 0), (0, 10), (10, 1000), (1000, 1001), (1001, 3995), (0, 0), (3995, 4000)]]
    assert out.check("sums").cpu().tolist() == want


@pytest.mark.parametrize("t", ["f32", "f64"])
def test_a_tiled_segment_changes_no_other(t):
    """Segments above 64 KiB are cut into tiles by a second launch."""
    eb = 4 if t == "f32" else 8
    L = np.array([4096 // eb + 1, 300, 65536 // eb, 7, 20000 // eb, 0, 33333 // eb, 200000 // eb], dtype=np.int64)
    off = inputs.offsets_from_lengths(L) + 1
    v = torch.from_numpy(inputs.normal(int(off[-1]), np.float32 if t == "f32" else np.float64)).cuda()
    got = []
    for n in (len(L), len(L) - 1):  # with the tiled last one, without
        s, m = torch.zeros(n, dtype=TD[t], device="cuda"), torch.zeros(n, dtype=TD[t], device="cuda")
        api.accr_segmented_reduce(v, off[:n + 1], [api.clause("add", s), api.clause("min", m)], flags=api.ACCR_SYNC)
        got.append((s[:len(L) - 1].cpu(), m[:len(L) - 1].cpu()))
    for a, b in zip(*got):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
