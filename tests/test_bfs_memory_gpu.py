"""The persistent search without memory for its bitmaps: cell by cell where they are
large, an error where they are not (an injected failure then reports as everywhere)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1412_1127_gb300 import api, inputs
from paper_1412_1127_gb300._native import ACCR_ENOMEM, AccrError

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_faults_left():
    yield
    api.accr_fault_inject(api.ACCR_FAULT_ALLOC, 0)


def maze(rows, cols):
    grid = (inputs.rng(47, rows).random((rows, cols)) < 0.8).astype(np.uint8)
    src = (rows // 2) * cols + cols // 2
    grid.flat[src] = 1
    return grid, src


def test_large_bitmaps_that_cannot_be_had():
    grid, src = maze(1500, 3000)
    want, wl = oracle.grid_bfs(grid, src)
    gt, dist = torch.from_numpy(grid).cuda(), torch.empty(1500, 3000, dtype=torch.int32, device="cuda")
    fresh = torch.cuda.Stream()
    torch.cuda.synchronize()
    for faults, launches in ((1, 2), (0, 1)):  # without, then with memory: the tiles again
        api.accr_fault_inject(api.ACCR_FAULT_ALLOC, faults)
        before = api.accr_launch_count()
        assert api.accr_grid_bfs(gt, src, dist, mode="persistent", stream=fresh) == wl
        assert api.accr_launch_count() - before == launches
        assert np.array_equal(dist.cpu().numpy(), want)
    assert api.accr_last_error() == ""


def test_other_failures_are_reported():
    for shape, faults in (((100, 100), 1), ((1500, 3000), 2)):
        grid, src = maze(*shape)
        gt, dist = torch.from_numpy(grid).cuda(), torch.empty(*shape, dtype=torch.int32, device="cuda")
        fresh = torch.cuda.Stream()
        torch.cuda.synchronize()
        api.accr_fault_inject(api.ACCR_FAULT_ALLOC, faults)
        with pytest.raises(AccrError) as e:
            api.accr_grid_bfs(gt, src, dist, mode="persistent", stream=fresh)
        assert e.value.code == ACCR_ENOMEM
        api.accr_fault_inject(api.ACCR_FAULT_ALLOC, 0)
        want, wl = oracle.grid_bfs(grid, src)
        assert api.accr_grid_bfs(gt, src, dist, mode="persistent", stream=fresh) == wl
        assert np.array_equal(dist.cpu().numpy(), want)
