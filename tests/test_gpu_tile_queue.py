"""The longest-first tile queue keeps the tiles' order among lists of equal length, whatever CTAs built it: the render
backward takes the tiles in that order, and its float sums follow it."""
import numpy as np
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _queue(n, sizes, tile, seed=0):
    rng = np.random.default_rng(seed)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    t = [f(np.concatenate([rng.normal(0, 0.5, (n, 3)), rng.uniform(0.2, 0.9, (n, 1))], 1)),
         f(np.concatenate([rng.normal(-4, 0.5, (n, 3)), rng.uniform(1, 4, (n, 1))], 1)), f(rng.normal(size=(n, 4))),
         f(rng.uniform(size=(n, 3)))]
    cams = [look_at((0.3 * k, -4.0, 0.2), (0, 0, 0), w, h) for k, (w, h) in enumerate(sizes)]
    rast = api.Rasterizer(n, cams, api.GESConfig(tile_w=tile[0], tile_h=tile[1], persistent=1))
    rast.preprocess(*t)
    rast.bin()
    bv = rast.bins_views(1)
    rg = bv["ranges"].cpu().numpy().astype(np.int64)
    return (rg[:, 1] - rg[:, 0]), bv["queue"].cpu().numpy()


# one CTA of the index (1,024 tiles), one more tile, many CTAs, several views, CTAs of 2,048 tiles
@pytest.mark.parametrize("n,sizes,tile", [(3000, [(256, 256)], (8, 8)), (3000, [(520, 128)], (8, 8)),
                                          (40000, [(1601, 1040)], (16, 8)),
                                          (9000, [(997, 661), (400, 300), (64, 8)], (8, 8)),
                                          (50, [(8192, 5000)], (8, 8))])
def test_equal_lengths_keep_the_tiles_order(n, sizes, tile):
    lens, queue = _queue(n, sizes, tile)
    np.testing.assert_array_equal(np.sort(queue), np.arange(lens.size))
    bucket = np.where(lens > 0, np.floor(4 * np.log2(lens + 1.0) + 1e-4), -1)[queue]
    assert (bucket[1:] <= bucket[:-1] + 1).all()  # longest first, up to the buckets of a quarter octave
    order = np.lexsort((np.arange(queue.size), lens[queue]))  # stable by length
    tiles, same = queue[order], lens[queue][order]
    assert (tiles[1:] > tiles[:-1])[same[1:] == same[:-1]].all()
