"""KNN lists where the two-pass search can go wrong: ties at the 16th distance (lattices, duplicates), fewer
centres near the query than 16 (outliers, the smallest clouds), axes with more cells than the grid's limit
(a long line), sparse and dense regions in one cloud. Distances are the kernel's own float32 operations, so
the lists, ordered by (distance, index), must equal brute force exactly."""
import pytest
import torch

from paper_2411_09156_gb300 import api

pytestmark = pytest.mark.gpu


def _brute(centres, queries):
    out = []
    ids = torch.arange(centres.shape[0], device="cuda", dtype=torch.int64)
    for q in queries.split(512):
        d = (q[:, None, 0] - centres[None, :, 0]) ** 2
        d = d + (q[:, None, 1] - centres[None, :, 1]) ** 2
        d = d + (q[:, None, 2] - centres[None, :, 2]) ** 2
        key = (d.contiguous().view(torch.int32).to(torch.int64) << 32) | ids
        out.append((torch.topk(key, 16, dim=1, largest=False, sorted=True).values & 0xFFFFFFFF).to(torch.int32))
    return torch.cat(out)


def _cloud(name, g):
    r = lambda *s: torch.rand(*s, generator=g, device="cuda")
    if name == "lattice":
        ax = torch.arange(18.0, device="cuda")
        return torch.cat([torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3), r(5832, 1)], 1)
    if name == "plane-lattice":
        ax = torch.arange(64.0, device="cuda")
        return torch.cat([torch.stack(torch.meshgrid(ax, ax, torch.zeros(1, device="cuda"), indexing="ij"), -1).reshape(-1, 3),
                          r(4096, 1)], 1)
    if name == "duplicates":
        return r(500, 4).repeat(10, 1)
    if name == "coincident":
        return torch.ones(3000, 4, device="cuda")
    if name == "line":
        p = r(6000, 4)
        p[:, 1:3] = 0.25
        return p
    if name == "outliers":
        return torch.cat([0.01 * r(4000, 4), 3.0 + r(1500, 4), 80.0 * r(60, 4) - 40.0])
    return r(int(name), 4)


@pytest.mark.parametrize("name", ["lattice", "plane-lattice", "duplicates", "coincident", "line", "outliers", "16", "17",
                                  "65", "4099"])
def test_lists_equal_brute_force(name):
    g = torch.Generator(device="cuda").manual_seed(5)
    c = _cloud(name, g).contiguous()
    assert torch.equal(api.knn(c), _brute(c, c))
    # queries at centres, near them, on the box's edge and far outside
    pick = c[torch.randint(0, c.shape[0], (700,), generator=g, device="cuda")]
    q = torch.cat([pick[:200], pick[200:500] + 0.03 * torch.randn(300, 4, generator=g, device="cuda"),
                   pick[500:] + 5.0 * torch.randn(200, 4, generator=g, device="cuda")])
    q[:, 3] = 1.0
    q[::9, 3] = 0.0
    got, want = api.knn_points(c, q.contiguous()), _brute(c, q)
    want[q[:, 3] == 0.0] = -1
    assert torch.equal(got, want)
