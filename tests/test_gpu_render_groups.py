"""The forward walks each 8x4 pixel block as two 4x4 groups with their own splat lists. A pixel's value
must not depend on which of its block's and groups' pixels lie inside the view: a view cropped to its
first columns and rows renders the same bits as the full view there (the Jacobian clamp, which depends
on the view's size, is set out of reach)."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at, make_scene

pytestmark = pytest.mark.gpu


def _render(sc, cam, tile, persistent):
    cfg = api.GESConfig(tile_w=tile[0], tile_h=tile[1], persistent=persistent, jac_clamp=1e3, bg=(0.2, 0.4, 0.1))
    rast = api.Rasterizer(sc.n, [cam], cfg)
    rast.forward(*api.scene_tensors(sc))
    torch.cuda.synchronize()
    assert rast.sync_status() == 0
    return {k: rast.image(k, 0).clone() for k in ("color", "depth", "alpha", "normal", "t_final", "n_contrib")}


@pytest.mark.parametrize("tile", [(16, 16), (16, 8), (8, 8), (8, 32)])
@pytest.mark.parametrize("w,h", [(1, 1), (3, 2), (4, 4), (5, 3), (7, 9), (12, 5), (13, 17)])
def test_cropped_view_renders_the_full_views_bits(w, h, tile):
    sc = make_scene(3000, 17, "uniform", -1)
    full_cam = look_at((0.1, -3.2, 0.3), (0, 0, 0), 29, 23)
    full = _render(sc, full_cam, (16, 16), 0)
    crop = look_at((0.1, -3.2, 0.3), (0, 0, 0), 29, 23)
    crop.width, crop.height = w, h
    got = _render(sc, crop, tile, 1)
    assert int(full["n_contrib"][:h, :w].max()) > 0
    for k, g in got.items():
        assert torch.equal(g, full[k][..., :h, :w]), k
