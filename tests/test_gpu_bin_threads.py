"""Two host threads bin views of different size on streams of their own, again and again: each keeps its own lists, and
neither call disturbs the other's launches (the kernels' shared memory differs with the view)."""
import threading

import numpy as np
import pytest
import torch

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.scenes import look_at

pytestmark = pytest.mark.gpu


def _rast(n, w, h, tile, seed):
    rng = np.random.default_rng(seed)
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    t = [f(np.concatenate([rng.normal(0, 0.5, (n, 3)), rng.uniform(0.2, 0.9, (n, 1))], 1)),
         f(np.concatenate([rng.normal(-6, 0.3, (n, 3)), rng.uniform(1, 4, (n, 1))], 1)), f(rng.normal(size=(n, 4))),
         f(rng.uniform(size=(n, 3)))]
    rast = api.Rasterizer(n, [look_at((0.0, -4.0, 0.0), (0, 0, 0), w, h)], api.GESConfig(tile_w=tile[0], tile_h=tile[1]))
    rast.preprocess(*t)
    rast.bin()
    rast.fixed_capacity = True  # no read-back of the count in the loop
    return rast, rast.bins_views(rast.last_instance_count)["entry"].clone()


def test_threads_with_views_of_different_size():
    # the large view's counters take 52,000 bytes of shared memory a CTA, the small view's 256
    work = [(_rast(700_000, 1600, 1040, (16, 8), 1), 1500), (_rast(2_000, 64, 64, (8, 8), 2), 15000)]
    torch.cuda.synchronize()
    errors = []

    def loop(rast, entries, reps):
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                for _ in range(reps):
                    rast.bin(stream)
            stream.synchronize()
            assert torch.equal(rast.bins_views(rast.last_instance_count)["entry"], entries)
        except BaseException as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=loop, args=(r, e, k)) for (r, e), k in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
