"""Clouds so large that most squared distances overflow to infinity: those centres tie and come by index, as brute force
in float32 orders them."""
import pytest
import torch

from paper_2411_09156_gb300 import api

pytestmark = pytest.mark.gpu


def _brute(c, q):
    d = (q[:, None, 0] - c[None, :, 0]) ** 2
    d = d + (q[:, None, 1] - c[None, :, 1]) ** 2
    d = d + (q[:, None, 2] - c[None, :, 2]) ** 2
    key = (d.contiguous().view(torch.int32).to(torch.int64) << 32) | torch.arange(c.shape[0], device="cuda")
    return (torch.sort(key, dim=1).values[:, :16] & 0xFFFFFFFF).to(torch.int32)


@pytest.mark.parametrize("clusters,per", [(40, 5), (300, 1), (7, 40), (16, 16)])
@pytest.mark.parametrize("scale", [1e19, 2e19, 4e19])
def test_overflowing_distances_tie_by_index(clusters, per, scale):
    g = torch.Generator(device="cuda").manual_seed(clusters)
    mid = 2.0 * torch.rand(clusters, 1, 4, generator=g, device="cuda") - 1.0
    c = (scale * (mid + 1e-3 * torch.randn(clusters, per, 4, generator=g, device="cuda"))).reshape(-1, 4)
    c = c[torch.randperm(c.shape[0], generator=g, device="cuda")].contiguous()
    assert torch.equal(api.knn(c), _brute(c, c))
    q = c[::3].clone()
    q[:, :3] *= 0.99
    q[:, 3] = 1.0
    assert torch.equal(api.knn_points(c, q), _brute(c, q))
