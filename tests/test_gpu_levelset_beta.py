"""Neighbours that the level-set march may not leave out by their exponent at the ray's closest approach: with beta < 0 the
falloff rises away from the centre. Steep ones (large beta) without a term give the bits of no neighbour at all."""
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _points(others_opacity, centre, lscale, beta):
    g = torch.Generator().manual_seed(3)
    n, w = 16, 240
    pos = torch.zeros(n, 4)
    pos[:, 3] = others_opacity
    pos[0, 3] = 0.9
    pos[1:, :3] = torch.tensor(centre) + 0.01 * torch.randn(n - 1, 3, generator=g)
    lsb = torch.full((n, 4), float(lscale))
    lsb[0, :3] = -1.5
    lsb[:, 3] = beta
    lsb[0, 3] = 2.0
    quat = torch.randn(n, 4, generator=g)
    cam = look_at((0.0, -3.0, 0.0), (0, 0, 0), w, w)
    depth, alpha = torch.full((w * w,), 3.0), torch.ones(w * w)
    at = torch.tensor([y * w + x for y in range(117, 123) for x in range(117, 123)], dtype=torch.int32)
    pix = torch.stack([torch.zeros_like(at), at], 1)
    cu = lambda t: t.contiguous().cuda()
    return api.levelset(cu(pos), cu(lsb), cu(quat), [cam], cu(depth), cu(alpha), cu(pix), n_steps=17)


def test_negative_beta():
    # beta -2: P = 1 / Q, beyond 250 at the centre, 6 at the ends of the march
    a, b = _points(0.99, (0.0, 0.0, 0.0), 0.7, -2.0), _points(0.0, (0.0, 0.0, 0.0), 0.7, -2.0)
    assert (b[:, 7] == 1).all()
    assert (a[:, 6] != b[:, 6]).all()  # every ray crosses the level elsewhere


@pytest.mark.parametrize("beta", [8.0, 20.0, 20.5, 40.0])
def test_steep_neighbours_without_a_term(beta):
    a, b = _points(0.99, (0.35, 0.0, 0.1), -3.0, beta), _points(0.0, (0.35, 0.0, 0.1), -3.0, beta)
    assert (b[:, 7] == 1).all()
    assert torch.equal(a, b)
