"""Long tile lists at the limits of their split by depth: the shortest that is split and the longest, depths that fill the
segments evenly, crowd into part of the range (beside one far splat, or as a steep density), or cannot be split."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _depths(n, kind, g):
    u = torch.rand(n, generator=g, device="cuda")
    if kind == "even":
        return 0.1 * u
    if kind == "steep":  # half of them in a hundredth of the range
        return 0.1 * u ** 6
    if kind == "two-heaps":
        return 0.1 * torch.where(u < 0.5, 0.01 * u, 0.99 + 0.01 * u)
    if kind == "far":
        y = 0.05 * u
        y[n // 3] = 700.0
        return y
    # a heap of equal depths, too many for a segment, in an even list
    y = 0.1 * u
    y[: min(n // 2, 6000)] = 0.05
    return y


@pytest.mark.parametrize("kind", ["even", "steep", "two-heaps", "far", "heap"])
@pytest.mark.parametrize("n", [8191, 8192, 8193, 9217, 12_345, 16_385, 50_001, 131_071, 131_072, 131_073])
def test_split_lists(n, kind):
    g = torch.Generator(device="cuda").manual_seed(n)
    cam = look_at((0.0, -4.0, 0.0), (0, 0, 0), 640, 512)
    pos = torch.zeros(n, 3, device="cuda")
    pos[:, 1] = _depths(n, kind, g)
    z = 4.0 + pos[:, 1]
    # two tiles' middles beside the image's centre, which is a tile corner: two long lists side by side
    side = torch.where(torch.arange(n, device="cuda") % 3 == 0, -1.0, 1.0) if n > 30_000 else torch.ones(n, device="cuda")
    pos[:, 0] = side * z * (8.0 / cam.fx)
    pos[:, 2] = z * (8.0 / cam.fy)
    lsb = torch.full((n, 4), -8.0, device="cuda")
    lsb[:, 3] = 2.0
    quat = torch.nn.functional.normalize(torch.randn(n, 4, generator=g, device="cuda"), dim=1)
    t = [torch.cat([pos, torch.full_like(z[:, None], 0.3)], 1), lsb, quat, torch.rand(n, 3, generator=g, device="cuda")]
    rast = api.Rasterizer(n, [cam], api.GESConfig())
    rast.preprocess(*[x.contiguous() for x in t])
    rast.bin()
    bv = rast.bins_views(n)
    assert rast.last_instance_count == n < 512 * bv["n_tiles"]  # not in depth slabs
    rg = bv["ranges"].to(torch.int64)
    lens = rg[:, 1] - rg[:, 0]
    assert int(lens.sum()) == n and int((lens > 0).sum()) == (2 if n > 30_000 else 1)
    entry, tile = bv["entry"].to(torch.int64), bv["tile"].to(torch.int64)
    assert torch.equal(torch.sort(entry).values, torch.arange(n, device="cuda"))
    key = (rast.proj_views()["binrec"][entry, 3].to(torch.int64) << 32) | entry
    same = tile[1:] == tile[:-1]
    assert (key[1:] > key[:-1])[same].all() and int((~same).sum()) == (1 if n > 30_000 else 0)
    assert torch.equal(torch.bincount(tile, minlength=lens.numel()), lens)
    assert rast.sync_status() == 0
