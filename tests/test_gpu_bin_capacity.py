"""Lists beyond the capacity: kept are the first instances of all views in the order of (float32 depth, entry, tile),
each tile's in depth order, and nothing depends on the run. Splats of one tile, of a box of at most 32 tiles and of
larger boxes; depths that spread and that are all equal; one dense tile (depth slabs); capacities from none to one
less than needed, among them those that cut inside an entry."""
import numpy as np
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu

CASES = {  # n, spread, log-scale, depth, views, tile
    "small": (400, 0.5, -3.5, "spread", [(96, 64), (61, 130)], (8, 8)),
    "large-boxes": (300, 0.6, -0.5, "spread", [(203, 131), (77, 90), (64, 64)], (8, 8)),
    "equal-depth": (700, 0.5, -2.0, "equal", [(160, 120)], (16, 8)),
    "equal-depth-large": (60, 0.5, 0.5, "equal", [(320, 240)], (8, 8)),
    "one-tile": (9000, 0.05, -4.0, "spread", [(16, 16), (16, 16)], (16, 16)),
    "many": (120_000, 0.5, -5.0, "spread", [(403, 301), (640, 400)], (16, 8)),
}


def _splats(n, spread, lscale, depth):
    rng = np.random.default_rng(n)
    pos = rng.uniform(-spread, spread, (n, 3))
    if depth == "equal":
        pos[:, 1] = 0.0
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    return [f(np.concatenate([pos, rng.uniform(0.1, 0.9, (n, 1))], 1)),
            f(np.concatenate([rng.normal(lscale, 0.4, (n, 3)), rng.uniform(1, 4, (n, 1))], 1)), f(rng.normal(size=(n, 4))),
            f(rng.uniform(size=(n, 3)))]


@pytest.mark.parametrize("persistent", [0, 1])
@pytest.mark.parametrize("name", CASES)
def test_nearest_instances_are_kept(name, persistent):
    n, spread, lscale, depth, sizes, tile = CASES[name]
    t = _splats(n, spread, lscale, depth)
    # every camera looks along +y: equal y is equal depth
    cams = [look_at((0.0, -4.0, 0.0), (0, 0, 0), w, h) for w, h in sizes]
    cfg = api.GESConfig(tile_w=tile[0], tile_h=tile[1], persistent=persistent)
    full = api.Rasterizer(n, cams, cfg)
    full.forward(*t)
    m = full.last_instance_count
    bv = full.bins_views(m)
    ftile, entry = bv["tile"].cpu().numpy().astype(np.int64), bv["entry"].cpu().numpy().astype(np.int64)
    key = full.proj_views()["binrec"].cpu().numpy()[:, 3].view(np.uint32)[entry]
    near = np.lexsort((ftile, entry, key))  # the order in which instances are kept
    for cap in sorted({0, 1, 97, m // 7, m // 3, m // 3 + 1, m // 2, m - m // 10, m - 200, m - 1}):
        if cap < 0 or cap >= m:
            continue
        short = api.Rasterizer(n, cams, cfg, capacity=cap)
        short.forward(*t)
        kept = int(short.bins[:4].view(torch.int32).item())  # what the buffer holds, rounded up to its alignment
        assert min(cap, m) <= kept <= m
        want = near[:kept]
        want = want[np.lexsort((entry[want], key[want], ftile[want]))]
        short.capacity = kept  # (the same layout: the buffer is as large for all capacities up to what it holds)
        sv = short.bins_views(kept)
        np.testing.assert_array_equal(sv["entry"].cpu().numpy(), entry[want])
        np.testing.assert_array_equal(sv["tile"].cpu().numpy(), ftile[want])
        rg = sv["ranges"].cpu().numpy()
        np.testing.assert_array_equal(rg[:, 1] - rg[:, 0], np.bincount(ftile[want], minlength=bv["n_tiles"]))
        assert short.sync_status() == (2 if kept < m else 0)
