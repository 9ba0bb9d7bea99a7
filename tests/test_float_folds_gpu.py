"""Float folds on the pipes they run on: floats summed into a double by anchored
extraction, compensated sums with TwoSum, max and min in hardware order."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_1412_1127_gb300 import api, inputs
from tolerances import same_bits

pytestmark = pytest.mark.gpu

WIDE_KINDS = ["normal", "scales", "cancel", "tiny", "subnormal", "huge", "zeros", "minus_zeros", "sparse", "inf", "nan"]


def wide_values(kind, n):
    g = np.random.default_rng(n + len(kind))
    x = g.standard_normal(n).astype(np.float32)
    if kind == "scales":
        x = (x * np.exp2(g.uniform(-60, 60, n))).astype(np.float32)
    elif kind == "cancel":
        x[1::2] = -x[0:-1:2][: x[1::2].size]
    elif kind == "tiny":       # about the smallest magnitude the anchored sum takes (2^-70)
        x = (x * np.exp2(np.float32(-69))).astype(np.float32)
    elif kind == "subnormal":
        x = (x * np.exp2(np.float32(-140))).astype(np.float32)
    elif kind == "huge":       # about the largest (2^120) and the largest finite float
        x = (np.sign(x) * np.exp2(g.integers(116, 127, n))).astype(np.float32)
        x[:: 37] = np.finfo(np.float32).max
    elif kind in ("zeros", "minus_zeros"):
        x[:] = 0.0 if kind == "zeros" else -0.0
    elif kind == "sparse":
        x[g.random(n) < 0.97] = 0.0
    elif kind in ("inf", "nan"):
        x[n // 2] = np.inf if kind == "inf" else np.nan
    return x


@pytest.mark.parametrize("kind", WIDE_KINDS)
@pytest.mark.parametrize("n", [1, 31, 16384, 3 * 16384 + 5, (1 << 21) + 3])
@pytest.mark.parametrize("off", [0, 1])
def test_float_into_double_sum(kind, n, off):
    """Floats summed into a double: chunks of 32 go through the anchored
    extraction, others through double additions.  A chunk loses at most
    2^-54 of its largest value and every double addition rounds once, so the
    sum stays within (adds on one path) 2^-53 sum|x|; a chunk, a warp, a CTA
    and a grid tree make fewer than 128 of them per thread at these sizes."""
    x = wide_values(kind, n)
    t = torch.from_numpy(np.concatenate([np.zeros(off, np.float32), x])).cuda()[off:]
    s = torch.empty(1, dtype=torch.float64, device="cuda")
    m = torch.empty(1, dtype=torch.float32, device="cuda")
    api.accr_reduce(t, [api.clause("add", s, init=-0.0), api.clause("max", m)], flags=api.ACCR_SYNC)
    got = s.item()
    if kind == "inf":
        assert got == math.inf
    elif kind == "nan":
        assert math.isnan(got)
    elif kind == "minus_zeros":
        assert got == 0.0 and math.copysign(1.0, got) == -1.0
    else:
        want = math.fsum(x.astype(np.float64))
        bound = 128 * 2.0 ** -53 * math.fsum(np.abs(x.astype(np.float64)))
        assert abs(got - want) <= bound, (got, want)
    if kind != "nan":
        assert same_bits(m.cpu().numpy()[0], oracle.reduce(x, "max", "f32"))


@pytest.mark.parametrize("n", [5, 4096, 65543, (1 << 22) + 1])
def test_compensated_sum_with_range(n):
    """Sum, max and min of floats in one pass, signed zeros among the extremes."""
    x = inputs.normal(n, np.float32, salt=n % 11)
    x[:: 3] = 0.0
    x[1:: 3] = -0.0
    for y in (x, np.where(x > 0, np.float32(-0.0), x), np.where(x < 0, np.float32(0.0), x)):
        y = np.ascontiguousarray(y.astype(np.float32))
        t = torch.from_numpy(y).cuda()
        s, hi, lo = (torch.empty(1, dtype=torch.float32, device="cuda") for _ in range(3))
        api.accr_reduce(t, [api.clause("add", s), api.clause("max", hi), api.clause("min", lo)],
                        flags=api.ACCR_COMPENSATED | api.ACCR_SYNC)
        assert same_bits(hi.cpu().numpy()[0], oracle.reduce(y, "max", "f32"))
        assert same_bits(lo.cpu().numpy()[0], oracle.reduce(y, "min", "f32"))
        want = math.fsum(y.astype(np.float64))
        # two roundings of the result and a second-order term
        assert abs(s.item() - want) <= 2.0 ** -23 * abs(want) + 2.0 ** -40 * math.fsum(np.abs(y.astype(np.float64)))
