"""The persistent search picks its form by the grid's shape: bit tiles in one launch, or
cell by cell (a set-up launch and the search) where most of a tile would stay empty."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from paper_1412_1127_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def search(grid, src, shape):
    dist = guarded(shape, torch.int32, 12345)
    before = api.accr_launch_count()
    levels = api.accr_grid_bfs(grid, src, dist.t, mode="persistent")
    return dist.check("dist").cpu().numpy(), levels, api.accr_launch_count() - before


@pytest.mark.parametrize("rows,cols,tiles", [(1000000, 1, False), (200000, 8, False), (100000, 3, False), (20000, 1, True),
                                             (20000, 40, True), (1000000, 40, True), (1, 200000, True), (8, 100000, True),
                                             (1024, 1024, True)])
def test_long_strips(rows, cols, tiles):
    """Open strips closed off 700 cells either way from the source: every level is known."""
    grid = torch.ones(rows, cols, dtype=torch.uint8, device="cuda")
    reach = min(700, max(rows, cols) // 2 - 1)
    if rows >= cols:
        grid[rows // 2 + reach] = 0
        grid[rows // 2 - reach] = 0
    else:
        grid[:, cols // 2 + reach] = 0
        grid[:, cols // 2 - reach] = 0
    r, c = rows // 2, cols // 2
    dist, levels, launches = search(grid, r * cols + c, (rows, cols))
    y, x = np.arange(rows)[:, None], np.arange(cols)[None, :]
    want = np.abs(y - r) + np.abs(x - c)
    want[(np.abs(y - r) if rows >= cols else np.abs(x - c)) + 0 * want >= reach] = -1
    assert np.array_equal(dist, want)
    assert levels == int(want.max()) + 1
    assert launches == (1 if tiles else 2)


@pytest.mark.parametrize("rows,cols", [(60000, 2), (90000, 5), (150000, 17)])
def test_tall_mazes(rows, cols):
    g = inputs.rng(43, rows)
    grid = (g.random((rows, cols)) < 0.9).astype(np.uint8)
    grid[rows // 2 - 40:rows // 2 + 40] = 1
    src = (rows // 2) * cols
    want, wl = oracle.grid_bfs(grid, src)
    dist, levels, _ = search(torch.from_numpy(grid).cuda(), src, (rows, cols))
    assert levels == wl and np.array_equal(dist, want)
