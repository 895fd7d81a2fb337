"""The reported number of binning launches at the sides of each rule (a count only: nothing is launched)."""
import pytest

from paper_2411_09156_gb300.batch import binning_launches


@pytest.mark.parametrize("n,sizes,tile,capacity,launches", [
    (0, [(64, 64)], (16, 16), 10, 3),
    (4096, [(800, 800)], (16, 16), 1 << 20, 6),
    (4097, [(800, 800)], (16, 16), 1 << 20, 7),
    (16385, [(800, 800)], (16, 16), 1 << 20, 9),
    (16385, [(800, 800)], (16, 16), 4096, 6),
    # 512 entries a tile: 2,500 tiles
    (512 * 2500 - 1, [(800, 800)], (16, 16), 1 << 24, 9),
    (512 * 2500, [(800, 800)], (16, 16), 1 << 24, 10),
    (512 * 2500, [(800, 800), (800, 801)], (16, 16), 1 << 24, 9),
    # as dense, but two counters for each of 13,000 tiles do not fit: no split by depth, no depth-range pass
    (7_000_000, [(1600, 1040)], (16, 8), 1 << 26, 9),
    # 11,264 tiles do
    (7_000_000, [(2048, 704)], (16, 8), 1 << 26, 10),
])
def test_launch_count(n, sizes, tile, capacity, launches):
    assert binning_launches(n, sizes, *tile, capacity) == launches
