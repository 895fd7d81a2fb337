"""The GSR sample kernel copies a warp's neighbour records slot by slot through shared memory and adds a
neighbour's gradient with vector reductions. A sample's values must not depend on its place in a warp, on
the samples beside it, or on where invalid entries stand in its list; and the gradient of a set of samples
is the sum of its parts."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import make_scene

pytestmark = pytest.mark.gpu


def _inputs(n=700, seed=4):
    t = api.scene_tensors(make_scene(n, seed, "object", -1))
    g = torch.Generator().manual_seed(seed)
    return t, api.knn(t[0]), g


@pytest.mark.parametrize("m", [1, 31, 32, 33, 127, 129, 1000])
def test_samples_do_not_depend_on_their_place(m):
    t, nb, g = _inputs()
    splat = torch.randint(0, 700, (m,), generator=g).int()
    splat[::7] = torch.tensor([-1, 700, 2 ** 30], dtype=torch.int32).repeat(m)[: splat[::7].numel()]
    z = torch.randn(m, 3, generator=g)
    a = api.gsr(*t[:3], nb, splat.cuda(), z.cuda(), per_sample=True)
    p = torch.randperm(m, generator=g)
    b = api.gsr(*t[:3], nb, splat[p].contiguous().cuda(), z[p].contiguous().cuda(), per_sample=True)
    ok = ((splat >= 0) & (splat < 700))[p]
    assert torch.equal(a["sample_out"][p.cuda()][ok.cuda()], b["sample_out"][ok.cuda()])
    for k in ("g_pos_op", "g_lscale_beta", "g_quat"):
        # the same float32 terms added in another order: a splat's at most 17 (m + 1) terms, each rounded once
        tol = 1e-5 * float(a[k].abs().max())
        assert float((a[k] - b[k]).abs().max()) <= tol, k


def test_invalid_list_entries_are_skipped_wherever_they_stand():
    t, nb, g = _inputs()
    m = 700
    splat, z = torch.arange(m, dtype=torch.int32).cuda(), torch.randn(m, 3, generator=g).cuda()
    head = nb.clone()
    head[:, 9:] = -1
    spread = torch.full_like(nb, -1)
    spread[:, [1, 2, 3, 5, 7, 8, 11, 12, 15]] = nb[:, :9]
    spread[:, 4] = m  # one past the last splat
    a, b = (api.gsr(*t[:3], l.contiguous(), splat, z, per_sample=True) for l in (head, spread))
    assert torch.equal(a["sample_out"][:, :7], b["sample_out"][:, :7])
    assert torch.equal(a["losses"], b["losses"])
    none = api.gsr(*t[:3], torch.full_like(nb, -1), splat, z)
    assert all(float(none[k].abs().max()) == 0.0 for k in ("losses", "g_pos_op", "g_lscale_beta", "g_quat"))


def test_gradient_is_the_sum_of_its_parts():
    t, nb, g = _inputs()
    m = 600
    splat, z = torch.randint(0, 700, (m,), generator=g).int().cuda(), torch.randn(m, 3, generator=g).cuda()
    whole = api.gsr(*t[:3], nb, splat, z)
    parts = [(0, 1), (1, 34), (34, 290), (290, m)]
    for k in ("losses", "g_pos_op", "g_lscale_beta", "g_quat"):
        s = sum((b - a) * api.gsr(*t[:3], nb, splat[a:b].contiguous(), z[a:b].contiguous())[k].double() for a, b in parts)
        # float32 sums of the same terms, scaled by 1 / m in float32: a few ulp of the largest value
        assert float((whole[k].double() * m - s).abs().max()) <= 1e-5 * float(s.abs().max()), k
