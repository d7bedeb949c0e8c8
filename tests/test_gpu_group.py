"""Grouping of a small batch by one cluster of blocks: batch sizes around the cluster's ranges and
its limit, material counts around two per thread and the limit, and materials out of range, against
the unsorted schedule (which groups nothing), bit for bit."""
import numpy as np
import pytest

from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 4097, 8191, 8192, 8193, 20000])
@pytest.mark.parametrize("n_mats", [1, 2, 1023, 1025, 2048, 2049])
def test_grouped_equals_unsorted(n, n_mats):
    import torch
    nets = W.random_materials(min(n_mats, 16), 4, 12, 0.3, seed=8)
    mats = [nets[m % len(nets)] for m in range(n_mats)]
    pts = W.points_uniform(n, seed=n, n_mats=n_mats)
    rng = np.random.default_rng(n)
    for k in ("u", "v"):
        pts[k] = np.round(pts[k] * 32) / 32
    bad = rng.random(n) < 0.05
    pts["mat"] = np.where(bad, n_mats + rng.integers(0, 3, n), pts["mat"]).astype(np.uint32)
    d, res = P.points_to_device(pts), []
    for flags in (0, P.PMC_UNSORTED):
        c = P.Cache(mats, 4096, 8)
        c.set_schedule(flags)
        out = []
        for _ in range(2):
            rgb = torch.full((3, n), 7.0, device="cuda")
            hits = torch.full((n,), 99, dtype=torch.int16, device="cuda")
            c.eval_batch(d, rgb, hits)
            out.append((rgb, hits))
        try:
            c.sync()
        except P.PmcError as e:   # materials out of range are reported
            assert bad.any() and e.status == P.PMC_ERR_INVALID_ARG
        out = [(r.cpu().numpy(), h.cpu().numpy()) for r, h in out]
        res.append((out, c.stats(), c.table()))
    for (r0, h0), (r1, h1) in zip(res[0][0], res[1][0]):
        assert np.array_equal(r0, r1) and np.array_equal(h0, h1)
        assert not r0[:, bad].any() and not h0[bad].any()
    s0, s1 = res[0][1], res[1][1]
    assert all(s0[k] == s1[k] for k in ("points", "bad_points", "lookups", "hits", "inserted", "batches"))
    for x, y in zip(res[0][2], res[1][2]):
        assert np.array_equal(x, y)
