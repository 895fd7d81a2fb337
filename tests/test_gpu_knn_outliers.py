"""Centres far from all others in a long thin cloud: exact lists, and no time spent on rows of cells outside the grid."""
import pytest
import torch

from paper_2411_09156_gb300 import api

pytestmark = pytest.mark.gpu


def _brute(c):
    d = (c[:, None, 0] - c[None, :, 0]) ** 2
    d = d + (c[:, None, 1] - c[None, :, 1]) ** 2
    d = d + (c[:, None, 2] - c[None, :, 2]) ** 2
    key = (d.contiguous().view(torch.int32).to(torch.int64) << 32) | torch.arange(c.shape[0], device="cuda")
    return (torch.topk(key, 16, dim=1, largest=False, sorted=True).values & 0xFFFFFFFF).to(torch.int32)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_line_with_outliers(axis):
    g = torch.Generator(device="cuda").manual_seed(3)
    c = torch.full((6000, 4), 0.25, device="cuda")
    c[:, axis] = torch.rand(6000, generator=g, device="cuda")
    c[100:, axis] *= 0.001  # 100 centres over 2,048 cells, the others in the first few
    assert torch.equal(api.knn(c), _brute(c))
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    api.knn(c)
    b.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(b) < 60.0  # ms: some 3, 300 with rings over rows that are not there
