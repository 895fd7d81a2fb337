"""The preprocess takes 32 splats of one view a warp, or 16 of two where a splat's coefficients are long (float32
SH2 and SH3); an odd last view is taken alone. Every entry's records must be the ones that a call with its view
alone writes, bit for bit, whole and in ranges that start anywhere."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at, make_scene

pytestmark = pytest.mark.gpu


def _records(rast, n_views, v, n):
    lay = api.ges_get_layout(n, n_views, rast.cams_c, rast.cfg_c, 1)
    rec = rast.proj[lay.proj_records:lay.proj_records + 64 * n * n_views].view(n_views, n, 64)[v]
    binrec = rast.proj[lay.proj_binrec:lay.proj_binrec + 32 * n * n_views].view(n_views, n, 32)[v]
    return rec.clone(), binrec.clone()


@pytest.mark.parametrize("sh,storage", [(-1, 0), (1, 0), (2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("views", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("n", [1, 17, 33, 1000])
def test_records_equal_those_of_single_views(n, views, sh, storage):
    t = list(api.scene_tensors(make_scene(n, 11, "uniform", sh)))
    if storage:
        t[3] = t[3].to(torch.float16)
    cams = [look_at((0.3 * v - 0.5, -3.0, 0.2 * v), (0, 0, 0), 64 + 8 * v, 48 + 4 * v) for v in range(views)]
    cfg = api.GESConfig(sh_degree=sh, color_storage=storage)
    whole, parts = api.Rasterizer(n, cams, cfg), api.Rasterizer(n, cams, cfg)
    whole.preprocess(*t)
    cuts = sorted({0, min(n, 5), n // 2, n})
    for a, b in zip(cuts, cuts[1:]):
        parts.preprocess_range(a, b - a, *t)
    total = 0
    for v, cam in enumerate(cams):
        one = api.Rasterizer(n, [cam], cfg)
        one.preprocess(*t)
        total += api.ges_instance_count(one.proj)
        for want, got, ranged in zip(_records(one, 1, 0, n), _records(whole, views, v, n),
                                     _records(parts, views, v, n)):
            assert torch.equal(want, got) and torch.equal(want, ranged), v
    assert total == api.ges_instance_count(whole.proj) == api.ges_instance_count(parts.proj) and (n < 17 or total > 0)
