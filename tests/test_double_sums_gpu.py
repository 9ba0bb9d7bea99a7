"""Sums of doubles over every entry point: what a chunk summed in integer block
floating point cannot hold goes through double additions."""
import math

import numpy as np
import pytest
import torch

from paper_1412_1127_gb300 import api

pytestmark = pytest.mark.gpu

INF, NAN = math.inf, math.nan
# planted values and what IEEE additions in any order make of them and finite others
PLANTED = [((INF,), INF), ((-INF,), -INF), ((INF, -INF), NAN), ((INF, -1e300), INF), ((INF, -1.5e308), INF),
           ((NAN,), NAN), ((INF, INF), INF)]


def planted(n, values, seed):
    g = np.random.default_rng(seed)
    x = g.standard_normal(n)
    x[g.permutation(n)[:len(values)]] = values[:n]
    return x


def same(got, want):
    return math.isnan(got) if math.isnan(want) else got == want


@pytest.mark.parametrize("values,want", PLANTED)
@pytest.mark.parametrize("n", [2, 3, 100, 511, 513, 2100, 9001, 40000, 70001, 300007])
def test_infinities_and_nan(n, values, want):
    """Short stretches (one partial round) and long ones, alone and beside a maximum."""
    xs = [planted(n, values, seed) for seed in (1, 2, 3)]
    flat = torch.from_numpy(np.concatenate(xs)).cuda()
    off = np.arange(4, dtype=np.int64) * n
    z = lambda: torch.zeros(3, dtype=torch.float64, device="cuda")
    got = {}
    s = z()
    for i in range(3):
        api.accr_reduce(flat[off[i]:off[i + 1]], [api.clause("add", s[i:i + 1])])
    got["region"] = s
    s, m = z(), z()
    for i in range(3):
        api.accr_reduce(flat[off[i]:off[i + 1]], [api.clause("max", m[i:i + 1]), api.clause("add", s[i:i + 1])])
    got["region, sum and max"] = s
    for name, others in (("alone", 0), ("with min", 1), ("with two", 2)):
        for entry in ("rows", "segments"):
            s = z()
            cl = [api.clause("add", s)] + [api.clause(op, z()) for op in ("min", "max")[:others]]
            if entry == "rows":
                api.accr_rowreduce(flat.view(3, n), cl)
            else:
                api.accr_segmented_reduce(flat, off, cl)
            got[entry + " " + name] = s
    s = z()
    api.accr_batch_reduce([(flat[off[i]:off[i + 1]], [api.clause("add", s[i:i + 1])], 0) for i in range(3)])
    got["batch"] = s
    torch.cuda.synchronize()
    bad = {k: v.tolist() for k, v in got.items() if not all(same(x, want) for x in v.tolist())}
    assert not bad, (want, bad)
