"""The level-set march leaves out neighbours whose terms are exactly 0 along the whole ray. Such a neighbour and one of
opacity 0 must give the same bits; one that matters must not be left out."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _points(others_opacity, offset, lscale, beta, steps):
    g = torch.Generator().manual_seed(3)
    n = 16
    pos = torch.zeros(n, 4)
    pos[:, 3] = others_opacity
    pos[0, 3] = 0.9
    pos[1:, 0] = offset + 0.3 * offset * torch.rand(n - 1, generator=g)
    pos[1:, 2] = 0.2 * offset * torch.randn(n - 1, generator=g)
    lsb = torch.full((n, 4), float(lscale))
    lsb[0, :3] = -1.5
    lsb[:, 3] = beta
    quat = torch.randn(n, 4, generator=g)
    cam = look_at((0.0, -3.0, 0.0), (0, 0, 0), 24, 24)
    depth, alpha = torch.full((576,), 3.0), torch.ones(576)
    pix = torch.stack([torch.zeros(576, dtype=torch.int32), torch.arange(576, dtype=torch.int32)], 1)
    cu = lambda t: t.contiguous().cuda()
    return api.levelset(cu(pos), cu(lsb), cu(quat), [cam], cu(depth), cu(alpha), cu(pix), n_steps=steps)


@pytest.mark.parametrize("steps", [2, 16, 17, 33])
@pytest.mark.parametrize("beta", [1.0, 2.0, 6.0])
def test_neighbours_without_a_term(beta, steps):
    # scales of e^-9 beside rays up to 1 away: exponents beyond float32's end along every ray
    gone = _points(0.99, 3.0, -9.0, beta, steps)
    assert torch.equal(gone, _points(0.0, 3.0, -9.0, beta, steps))
    # (two samples, both ends of the range, never bracket the level)
    assert steps == 2 or int(gone[:, 7].sum()) > 0
    # the same neighbours as wide as the first splat do change the points
    near = _points(0.99, 0.3, -1.5, beta, steps)
    assert steps == 2 or not torch.equal(near, _points(0.0, 0.3, -1.5, beta, steps))
