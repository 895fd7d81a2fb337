"""One long list that is not split by depth: a view with so many tiles that its entries are few for each, all of them in
one tile. Lengths on both sides of every sort class, lists of so many chunks that a warp (32) and a CTA (1,024) take
several each; depths that spread, that are equal, in clusters, and one far splat that puts all others into one
depth bucket."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _one_tile(n, depth, width, height, tile):
    g = torch.Generator(device="cuda").manual_seed(n)
    cam = look_at((0.0, -4.0, 0.0), (0, 0, 0), width, height)
    r = lambda *s: torch.rand(*s, generator=g, device="cuda")
    pos = torch.zeros(n, 3, device="cuda")
    if depth == "spread":
        pos[:, 1] = 0.1 * r(n) - 0.05
    elif depth == "clusters":
        pos[:, 1] = torch.randint(0, 3, (n,), generator=g, device="cuda") * 0.02 + \
            torch.randint(0, 2, (n,), generator=g, device="cuda") * 1e-6
    elif depth == "far":
        pos[:, 1] = 0.001 * r(n)
        pos[n // 2, 1] = 900.0
    # the middle of the tile beside the image's centre, which is a tile corner; the far splat on the same ray
    z = 4.0 + pos[:, 1]
    pos[:, 0] = z * (0.5 * tile / cam.fx)
    pos[:, 2] = z * (0.5 * tile / cam.fy)
    t = [torch.cat([pos, 0.3 + 0.0 * pos[:, :1]], 1), torch.full((n, 4), -8.0, device="cuda"),
         torch.nn.functional.normalize(torch.randn(n, 4, generator=g, device="cuda"), dim=1), r(n, 3)]
    t[1][:, 3] = 2.0
    rast = api.Rasterizer(n, [cam], api.GESConfig(tile_w=tile, tile_h=tile))
    rast.preprocess(*[x.contiguous() for x in t])
    rast.bin()
    return rast


def _check(rast, n):
    m = rast.last_instance_count
    bv = rast.bins_views(m)
    assert n < 512 * bv["n_tiles"]  # not split by depth
    lens = (bv["ranges"][:, 1] - bv["ranges"][:, 0]).to(torch.int64)
    assert m == n and int(lens.max()) == n and int(lens.sum()) == n  # one list
    entry = bv["entry"].to(torch.int64)
    assert torch.equal(torch.sort(entry).values, torch.arange(n, device="cuda"))
    key = (rast.proj_views()["binrec"][entry, 3].to(torch.int64) << 32) | entry
    assert (key[1:] > key[:-1]).all()  # by depth, then entry
    assert (bv["tile"] == bv["tile"][0]).all()
    assert rast.sync_status() == 0


@pytest.mark.parametrize("depth", ["spread", "equal", "clusters", "far"])
@pytest.mark.parametrize("n", [256, 257, 1024, 1025, 4096, 4097, 16384, 16385, 32769, 600_000])
def test_one_list(n, depth):
    _check(_one_tile(n, depth, 640, 512, 16), n)


@pytest.mark.parametrize("depth", ["spread", "equal", "far"])
def test_more_chunks_than_threads(depth):
    n = 17_000_000
    _check(_one_tile(n, depth, 2048, 2048, 8), n)
