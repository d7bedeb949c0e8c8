"""Batched misses of many cacheable nodes with few misses each: around the number of work items per node
from which a warp takes two, the same tables, counters and outputs as one miss per lane."""
import numpy as np
import pytest

from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [70000, 150000, 290000, 330000])   # 1 to 4 items of 32 misses per node
def test_pairs_equal_singles(n):
    import torch
    # equal short programs, so that the other line, 60 items per SM, is passed as well
    mats = W.random_materials(1, 60, 60, 0.2, 0) * 600
    first = W.points_uniform(3000, seed=1, n_mats=600)
    pts = W.points_uniform(n, seed=2, n_mats=600)
    res = []
    for flags in (0, P.PMC_ONE_POINT):
        c = P.Cache(mats, 1 << 18, 8)
        c.set_schedule(flags)
        for p in (first, pts):
            rgb = torch.empty((3, len(p["mat"])), device="cuda")
            hits = torch.empty(len(p["mat"]), dtype=torch.int16, device="cuda")
            c.eval_batch(P.points_to_device(p), rgb, hits)
        c.sync()
        res.append((rgb.cpu().numpy(), hits.cpu().numpy(), c.stats(), c.table()))
    a, b = res
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert a[2] == b[2]
    assert all(np.array_equal(x, y) for x, y in zip(a[3], b[3]))
