"""With one view the preprocess backward stages a warp's SH gradients in shared memory and stores them in runs
(SH degrees 2 and 3). The stored rows must not depend on how the splats fall into warps: ranges that start
anywhere, a last warp that is not full, and a gradient buffer that is not 16-byte aligned give the same bits
as one aligned call."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at, make_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sh", [-1, 0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 31, 33, 1000])
def test_gradient_rows_do_not_depend_on_ranges_or_alignment(n, sh):
    t = api.scene_tensors(make_scene(n, 7, "uniform", sh))
    rast = api.Rasterizer(n, [look_at((0.1, -3.0, 0.2), (0, 0, 0), 64, 48)], api.GESConfig(sh_degree=sh))
    rast.forward(*t)
    g = torch.Generator().manual_seed(n)
    rast.backward_screen(*[torch.randn(k * rast.P, generator=g).cuda() for k in (3, 1, 1, 3)])
    new = lambda: dict(g_pos_op=torch.empty_like(t[0]), g_lscale_beta=torch.empty_like(t[1]),
                       g_quat=torch.empty_like(t[2]), g_color=torch.full(t[3].shape, float("nan"), device="cuda"))
    whole = rast.preprocess_bwd(*t, new())
    assert torch.isfinite(whole["g_color"]).all() and (n < 31 or float(whole["g_color"].abs().max()) > 0)
    parts, cuts = new(), sorted({0, min(n, 5), n // 2, n})
    for a, b in zip(cuts, cuts[1:]):
        rast.preprocess_bwd_range(a, b - a, *t, parts)
    moved = new()
    flat = torch.full((t[3].numel() + 2,), 3.0, device="cuda")
    moved["g_color"] = flat[1:-1].view(t[3].shape)  # 4 bytes past an aligned address
    rast.preprocess_bwd(*t, moved)
    for k, w in whole.items():
        assert torch.equal(w, parts[k]) and torch.equal(w, moved[k]), k
    assert float(flat[0]) == 3.0 and float(flat[-1]) == 3.0
