"""Tile lists at the sizes where the list sort changes its way: a warp, a part or a whole CTA, one large CTA, chunks
with a merge; one list, many lists of mixed lengths; depths that spread, that are all equal (ties by entry), that
fall into a few clusters, and one far splat that puts all others into one depth bucket. The list must be
exactly the listed entries ordered by (float32 depth, entry)."""
import numpy as np
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _splats(n, depth, seed=0, spread=0.05, lscale=-1.0):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(-spread, spread, size=(n, 3))
    if depth == "equal":
        pos[:, 1] = 0.0
    elif depth == "clusters":
        pos[:, 1] = rng.integers(0, 3, n) * 0.5 + rng.integers(0, 2, n) * 1e-6
    elif depth == "far":
        pos[0, 1] = 900.0
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    return [f(np.concatenate([pos, np.full((n, 1), 0.5)], 1)),
            f(np.concatenate([np.full((n, 3), lscale), rng.uniform(1, 4, (n, 1))], 1)), f(rng.normal(size=(n, 4))),
            f(rng.uniform(size=(n, 3)))]


def _check(rast, n_views):
    m = rast.last_instance_count
    bv, pv = rast.bins_views(m), rast.proj_views()
    tile, entry = bv["tile"].cpu().numpy(), bv["entry"].cpu().numpy()
    rec = pv["binrec"].cpu().numpy()
    assert tile.size == m == rec[:, 2].sum()
    np.testing.assert_array_equal(np.bincount(entry, minlength=rec.shape[0]), rec[:, 2])  # each entry on all its tiles
    key = rec[entry, 3].view(np.uint32)
    order = np.lexsort((entry, key, tile))
    np.testing.assert_array_equal(order, np.arange(m))  # sorted by tile, depth, entry
    assert np.unique(tile.astype(np.int64) * rec.shape[0] + entry).size == m
    rg = bv["ranges"].cpu().numpy()
    lens = np.bincount(tile, minlength=rg.shape[0])
    np.testing.assert_array_equal(rg[:, 1] - rg[:, 0], lens)
    starts = np.concatenate([[0], np.cumsum(lens)[:-1]])
    np.testing.assert_array_equal(rg[:, 0], np.where(lens > 0, starts, 0))
    assert rast.sync_status() == 0
    return lens


@pytest.mark.parametrize("depth", ["spread", "equal", "clusters", "far"])
@pytest.mark.parametrize("n", [1, 31, 33, 255, 256, 257, 1023, 1025, 4095, 4096, 4097, 16384, 16385, 33000])
def test_one_list_of_every_class(n, depth):
    cam = look_at((0.0, -4.0, 0.0), (0, 0, 0), 16, 16)
    rast = api.Rasterizer(n, [cam], api.GESConfig(persistent=1))
    rast.forward(*_splats(n, depth))
    assert _check(rast, 1).max() >= n - 1  # (the far splat may miss the tile)


@pytest.mark.parametrize("tile", [(8, 8), (16, 8), (32, 8)])
def test_mixed_lists_views_and_capacity(tile):
    # a dense middle and sparse surroundings: lists of all classes at once, in two views of different size
    a, b = _splats(20000, "spread", 1, 0.05, -4.0), _splats(7001, "spread", 2, 1.5, -3.0)
    t = [torch.cat([x, y]) for x, y in zip(a, b)]
    cams = [look_at((0.0, -4.0, 0.0), (0, 0, 0), 203, 131), look_at((3.0, -2.0, 1.0), (0, 0, 0), 77, 90)]
    cfg = api.GESConfig(tile_w=tile[0], tile_h=tile[1], persistent=1)
    rast = api.Rasterizer(27001, cams, cfg)
    rast.forward(*t)
    lens = _check(rast, 2)
    assert lens.max() > 4096 and (lens == 0).any()
    queue = rast.bins_views(1)["queue"].cpu().numpy()
    np.testing.assert_array_equal(np.sort(queue), np.arange(lens.size))
    # longest first, up to the buckets of a quarter octave
    bucket = np.where(lens > 0, np.floor(4 * np.log2(lens + 1.0) + 1e-4), -1)[queue]
    assert (bucket[1:] <= bucket[:-1] + 1).all()
    # exactly enough capacity keeps every instance; one less reports it and keeps the ranges inside
    m = rast.last_instance_count
    exact = api.Rasterizer(27001, cams, cfg, capacity=m)
    exact.forward(*t)
    for k in ("color", "last", "n_contrib"):
        assert torch.equal(exact.out[k], rast.out[k])
    assert exact.sync_status() == 0
    short = api.Rasterizer(27001, cams, cfg, capacity=m - m // 3)
    short.forward(*t)
    assert short.sync_status() == 2
    rg = short.bins_views(1)["ranges"].cpu().numpy()
    assert (rg[:, 0] <= rg[:, 1]).all() and rg.max() <= m
