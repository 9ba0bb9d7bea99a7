"""The application patterns at the sizes and inputs where their forms change."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from paper_1412_1127_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,p", [((64, 1024), 0.7), ((65, 40), 0.7), ((64, 1025), 0.8), ((63, 3000), 0.75),
                                     ((129, 1), 1.0), ((4000, 33), 0.8), ((500, 1100), 0.62), ((2000, 2000), 0.7),
                                     ((31, 31), 0.0), ((1, 5000), 1.0), ((6000, 64), 0.9)])
def test_grid_bfs_tiles(shape, p):
    g = inputs.rng(33, shape[0] + shape[1])
    grid = (g.random(shape) < p).astype(np.uint8)
    for src in (0, shape[0] * shape[1] - 1, (shape[0] // 2) * shape[1] + shape[1] // 2):
        grid.flat[src] = 1
        want, wl = oracle.grid_bfs(grid, src)
        dist = guarded(shape, torch.int32, 12345)
        assert api.accr_grid_bfs(torch.from_numpy(grid).cuda(), src, dist.t, mode="persistent") == wl
        assert np.array_equal(dist.check("dist").cpu().numpy(), want)
    assert api.accr_grid_bfs(torch.from_numpy(grid).cuda(), -1, dist.t, mode="persistent") == 0
    assert bool((dist.t == -1).all())
