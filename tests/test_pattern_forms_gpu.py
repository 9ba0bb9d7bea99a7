"""The application patterns at the sizes and inputs where their forms change."""
import numpy as np
import pytest
import torch

import oracle
from guard import guarded
from paper_1412_1127_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def check_nearest(pts, qx, qy, k, what):
    for off in (0, 1):
        big = np.zeros((len(pts) + off, 2), dtype=np.float32)
        big[off:] = pts
        pt = torch.from_numpy(big).cuda()[off:]
        gi, gd = guarded((k,), torch.int64, -7), guarded((k,), torch.float32, -7)
        api.accr_nearest_k(pt, qx, qy, k, gi.t, gd.t, flags=api.ACCR_SYNC)
        wi, wd = oracle.nearest_k(pts, qx, qy, k)
        assert np.array_equal(gi.check("idx").cpu().numpy(), wi), (what, k, off)
        assert np.array_equal(gd.check("d2").cpu().numpy(), wd), (what, k, off)


@pytest.mark.parametrize("n", [15, 16, 63, 64, 65, 8191, 8192, 8193, 3 * 8192 + 1, 200003])
@pytest.mark.parametrize("k", [1, 2, 16])
def test_nearest_k_around_a_round(n, k):
    g = inputs.rng(31, n)
    check_nearest((g.random((n, 2), dtype=np.float32) * 100).astype(np.float32), 41.5, 58.25, k, n)


@pytest.mark.parametrize("k", [2, 10, 16])
@pytest.mark.parametrize("kind", ["one_warp_in_16", "clustered", "all_equal_but_few", "infinite", "mixed"])
def test_nearest_k_adversarial(kind, k):
    n = 300007
    g = inputs.rng(32, k)
    pts = (g.random((n, 2), dtype=np.float32) * 100).astype(np.float32)
    if kind == "one_warp_in_16":      # every near point in the same one of a CTA's 16 warps: a loose bound, many candidates
        i = np.arange(n)
        pts[(i // 64) % 16 != 3] += np.float32(500)
    elif kind == "clustered":         # the nearest thousand side by side
        pts[5000:6000] = 50 + g.random((1000, 2), dtype=np.float32)
    elif kind == "all_equal_but_few":
        pts[:] = np.float32(12.5)
        pts[[7, 299999, 150000]] = np.float32(50)
    elif kind == "infinite":          # all but three points infinitely far: they count, by index
        pts[:] = np.float32(3e38)
        pts[[11, 150001, n - 1]] = np.float32(49)
    else:                             # NaN among infinite ones
        pts[:] = np.float32(np.inf)
        pts[::2] = np.nan
        pts[[12, 4097]] = np.float32(51)
    check_nearest(pts, 50.0, 50.0, k, kind)


KEPT = 8 * 4 * 1024  # elements a CTA of the fused form keeps in registers


@pytest.mark.parametrize("n", [2, 3, 4, 4095, 4097, KEPT + 1, 152 * KEPT - 5, 152 * KEPT + 4099, 12345677])
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("in_place", [False, True])
def test_standardize_fused_forms(n, off, in_place):
    x = (inputs.normal(n, np.float32, salt=n % 13) * 3 + 5).astype(np.float32)
    xt = torch.from_numpy(np.concatenate([np.zeros(off, np.float32), x])).cuda()[off:]
    gy, gst = guarded((n,), torch.float32, float("nan")), guarded((2,), torch.float64, float("nan"))
    y = gy.t
    if in_place:
        gy.t.copy_(xt)
        xt = gy.t
    api.accr_standardize(xt, y, gst.t, flags=api.ACCR_SYNC)
    wy, (wm, wv) = oracle.standardize(x)
    mean, var = gst.check("stats").cpu().numpy()
    assert abs(mean - wm) <= 1e-9 * max(abs(wm), 1.0) and abs(var - wv) <= 1e-9 * wv
    got = gy.check("y").cpu().numpy()
    assert np.max(np.abs(got - wy) / np.maximum(np.abs(wy), 1.0)) <= 4e-6


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
