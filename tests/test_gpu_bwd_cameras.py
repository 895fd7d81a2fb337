"""The preprocess backward reads its cameras one by one (1 and 2 views) or packed (3 and more, tables of 4, 8, 16 and
32). With a screen-space gradient in one view alone the batched call must give that view's gradient: a lane that
reads another camera is off in the first digit. The single-view kernel may contract products otherwise: about 100
roundings of 2^-24, of terms up to 10 times the largest gradient, stay below 1e-4 of it."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at, make_scene

pytestmark = pytest.mark.gpu


def _screen_gradient(rast, n_views, n):
    at = api.ges_get_layout(n, n_views, rast.cams_c, rast.cfg_c, 1).proj_g2d
    return rast.proj[at:at + 64 * n * n_views].view(torch.float32).view(n_views, n, 16)


@pytest.mark.parametrize("views", [2, 3, 4, 7, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("n,sh", [(1, 3), (33, -1), (501, 3)])
def test_gradient_of_one_view_of_a_batch(n, sh, views):
    t = api.scene_tensors(make_scene(n, 5, "uniform", sh))
    cams = [look_at((0.1 * v - 0.8, -3.0 - 0.02 * v, 0.05 * v), (0, 0, 0), 64 + 8 * v, 48 + 4 * v)
            for v in range(views)]
    cfg = api.GESConfig(sh_degree=sh)
    batch = api.Rasterizer(n, cams, cfg)
    batch.preprocess(*t)
    new = lambda: dict(g_pos_op=torch.empty_like(t[0]), g_lscale_beta=torch.empty_like(t[1]),
                       g_quat=torch.empty_like(t[2]), g_color=torch.empty_like(t[3]))
    gen = torch.Generator().manual_seed(n + views)
    for v in sorted({0, views // 2, views - 1}):
        g = torch.randn((n, 16), generator=gen).cuda()
        one = api.Rasterizer(n, [cams[v]], cfg)
        one.preprocess(*t)
        _screen_gradient(one, 1, n)[0] = g
        screen = _screen_gradient(batch, views, n)
        screen.zero_()
        screen[v] = g
        want, got = one.preprocess_bwd(*t, new()), batch.preprocess_bwd(*t, new())
        for k, w in want.items():
            assert float(w.abs().max()) > 0, k
            assert float((w - got[k]).abs().max()) <= 1e-4 * float(w.abs().max()), (v, k)
