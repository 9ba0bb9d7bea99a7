"""accr_segmented_reduce at the limits of its lengths and offsets."""
import numpy as np
import pytest
import torch

from guard import guarded
from paper_1412_1127_gb300 import api

pytestmark = pytest.mark.gpu


def test_a_warp_folds_more_than_2_31_elements():
    """The warp-region limit is the caller's to set (accr_batch_tiling)."""
    n = (1 << 31) + 5
    v = torch.zeros(3 + n + 40, dtype=torch.int32, device="cuda")
    off = np.array([0, 3, 3 + n, 3 + n + 40], dtype=np.int64)
    marks = [0, 2, 3, 4096, 3 + (1 << 31) - 1, 3 + (1 << 31), 3 + n - 1, 3 + n, 3 + n + 39]
    for i, at in enumerate(marks):
        v[at] = 1 << i
    want = [sum(1 << i for i, at in enumerate(marks) if off[s] <= at < off[s + 1]) for s in range(3)]
    old = api.accr_batch_tiling(small_bytes=1 << 34)
    try:
        out = guarded((3,), torch.int64, 5)
        api.accr_segmented_reduce(v, off, [api.clause("add", out.t)], flags=api.ACCR_SYNC)
    finally:
        api.accr_batch_tiling(*old)
    assert out.check("sums").cpu().tolist() == want
