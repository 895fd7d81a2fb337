"""Queries that no distance bounds: points without coordinates (their lists stay empty), at infinity, or so far off that
every distance overflows (any 16 centres are as near as the others). They do not walk the whole grid."""
import pytest
import torch

from paper_2411_09156_gb300 import api

pytestmark = pytest.mark.gpu
M = 20_000


def _ms(f):
    f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    f()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b)


def _points(g, bad):
    q = torch.rand(M, 4, generator=g, device="cuda")
    q[:, 3] = 1.0
    for k in range(3):
        q[k::3, k] = bad
    return q


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf"), 1e30, -1e30])
def test_points_that_no_distance_bounds(bad):
    g = torch.Generator(device="cuda").manual_seed(1)
    q = _points(g, bad)
    c = torch.rand(3_200_000, 4, generator=g, device="cuda")
    got = api.knn_points(c, q)
    if bad != bad:
        assert (got == -1).all()
    else:
        assert ((got >= 0) & (got < c.shape[0])).all()
        assert (torch.sort(got, dim=1).values.diff(dim=1) > 0).all()  # 16 different centres
    # a second and more where each of the 20,000 queries reads every row of the grid, a tenth of this bound where it
    # ends at once
    assert _ms(lambda: api.knn_points(c, q)) < 250.0


def test_centres_without_coordinates():
    g = torch.Generator(device="cuda").manual_seed(2)
    c = torch.rand(50_000, 4, generator=g, device="cuda")
    c[7::1000, 1] = float("nan")
    got = api.knn(c)
    assert (got[7::1000] == -1).all()
    keep = torch.ones(50_000, dtype=torch.bool, device="cuda")
    keep[7::1000] = False
    ids = torch.nonzero(keep).squeeze(1).to(torch.int32)
    assert torch.equal(got[keep], ids[api.knn(c[keep].contiguous()).long()])
