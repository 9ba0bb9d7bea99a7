"""The forms of the row nest at the lengths where one gives way to another:
lane groups (1 to 32 lanes a row), a warp per row, segments (a warp or a CTA per
row), split rows.  Integer and extreme results bit-exact, float sums within
their worst-case bound, and a row alone gives the bits it gives in the matrix."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from paper_1412_1127_gb300 import api
from tolerances import same_bits

pytestmark = pytest.mark.gpu

TD = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32, "f64": torch.float64}
# bytes a row: every lane count's first and last length, the limits of the group (4 KiB),
# warp (16 KiB), segment (256 KiB) forms, each with a vector more or less
EDGES = [64, 128, 256, 512, 1024, 2048, 4096, 8192, 16384, 24576, 40960, 262144]
LENGTHS = sorted({max(1, e // 4 + d) for e in EDGES for d in (-5, -1, 0, 1, 4)} | {1, 2, 3, 5})


def matrix(rows, cols, t, pad, off):
    g = np.random.default_rng(rows * 131 + cols)
    big = g.integers(-(1 << 20), 1 << 20, size=(rows, cols + pad + off))
    big = (big.astype(np.float64) / (1 << 20)).astype(np.float32) if t == "f32" else big.astype(np.int32)
    return np.ascontiguousarray(big[:, off:off + cols]), torch.from_numpy(big).cuda()[:, off:off + cols]


def run(A, clauses, rows, flags=0):
    outs = [guarded((rows,), TD[acc], 9) for _, acc in clauses]
    api.accr_rowreduce(A, [api.clause(op, o.t) for (op, _), o in zip(clauses, outs)], flags=flags)
    return [o.check(op).cpu().numpy() for (op, _), o in zip(clauses, outs)]


def sum_bound(A, n):
    return n * 2.0 ** -24 * np.abs(A.astype(np.float64)).sum(1)


@pytest.mark.parametrize("cols", LENGTHS)
@pytest.mark.parametrize("pad,off", [(0, 0), (3, 1)])
def test_lengths_around_every_form(cols, pad, off):
    rows = 37
    I, It = matrix(rows, cols, "i32", pad, off)
    s, m = run(It, [("add", "i64"), ("max", "i32")], rows)
    assert np.array_equal(s, I.astype(np.int64).sum(1)) and np.array_equal(m, I.max(1))
    # a pair no kernel has fixed, its sum second: the generic fold, clauses in the caller's order
    x, a = run(It, [("bxor", "i32"), ("add", "i32")], rows)
    assert np.array_equal(x, np.bitwise_xor.reduce(I, axis=1)) and np.array_equal(a, I.sum(1, dtype=np.int32))
    F, Ft = matrix(rows, cols, "f32", pad, off)
    truth = F.astype(np.float64).sum(1)
    fs, fm = run(Ft, [("add", "f32"), ("min", "f32")], rows)
    assert same_bits(fm, F.min(1)) and np.all(np.abs(fs - truth) <= sum_bound(F, cols))
    wide, = run(Ft, [("add", "f64")], rows)
    assert np.all(np.abs(wide - truth) <= sum_bound(F, cols) * 2.0 ** -29)
    comp, = run(Ft, [("add", "f32")], rows, flags=api.ACCR_COMPENSATED)
    assert np.all(np.abs(comp - truth) <= 2.0 ** -23 * np.abs(truth) + sum_bound(F, cols) * 2.0 ** -16)
    for r in (0, 17, rows - 1):
        alone = run(Ft[r:r + 1], [("add", "f32"), ("min", "f32")], 1)
        assert same_bits(alone[0], fs[r:r + 1]) and same_bits(alone[1], fm[r:r + 1])


@pytest.mark.parametrize("cols", [4097, 5000, 9000])
def test_segment_rows_by_warp_and_by_cta(cols):
    """Enough rows for a warp each (a CTA each below that): the same bits."""
    rows = 24 * torch.cuda.get_device_properties(0).multi_processor_count
    F, Ft = matrix(rows, cols, "f32", 3, 1)
    many = run(Ft, [("add", "f32"), ("max", "f32")], rows)
    few = run(Ft[:rows // 2], [("add", "f32"), ("max", "f32")], rows // 2)
    assert same_bits(many[0][:rows // 2], few[0]) and same_bits(many[1][:rows // 2], few[1])
    assert same_bits(many[1], F.max(1))
    assert np.all(np.abs(many[0] - F.astype(np.float64).sum(1)) <= sum_bound(F, cols))
    D = torch.from_numpy(F[:100].astype(np.float64)).cuda()
    s, = run(D, [("add", "f64")], 100)
    assert np.all(np.abs(s - F[:100].astype(np.float64).sum(1)) <= sum_bound(F[:100], cols) * 2.0 ** -29)


@pytest.mark.parametrize("rows", [1, 31, 33, 5000])
def test_short_rows_every_operator(rows):
    I, It = matrix(rows, 21, "i32", 0, 0)
    I |= 1
    It = torch.from_numpy(I).cuda()
    for op in ["add", "mul", "max", "min", "band", "bor", "bxor", "land", "lor"]:
        got = run(It, [(op, "i64"), ("max", "i32"), (op, "i32")], rows)
        assert np.array_equal(got[0], oracle.rowreduce(I, op, "i64"))
        assert np.array_equal(got[2], oracle.rowreduce(I, op, "i32"))
