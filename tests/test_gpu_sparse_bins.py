"""Binned insert with few candidates in bins of fewer than 256 cells (passes after the first, whose
candidates are the few points not yet cached), every policy and table geometry that takes it, against
the oracle's sequential insert."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy,entries", [("binned", 4), ("binned", 8), ("replace", 8), ("keep", 16)])
@pytest.mark.parametrize("n_cells", [130, 500, 1500, 4099])
def test_sparse_bins_match_oracle(n_cells, policy, entries):
    import torch
    mats = W.random_materials(6, 20, 40, 0.3, seed=5)
    gpu = P.Cache(mats, n_cells, entries, flags={"binned": P.PMC_INSERT_BINNED, "replace": P.PMC_REPLACE_VISIBILITY,
                                                  "keep": 0}[policy])
    ref = O.Cache(mats, n_cells, entries, level=10, replacement=policy == "replace")
    n = 12001
    for p in range(4):
        pts = W.points_uniform(n, seed=p, n_mats=len(mats))
        for k in ("u", "v"):   # 900 texels, most of them seen in the first pass
            pts[k] = np.float32(np.floor(pts[k] * 30) / 30)
        if p:   # later passes: a few new texels
            new = np.random.default_rng(p).random(n) < 0.02
            pts["u"][new] = np.random.default_rng(p).random(int(new.sum())).astype(np.float32)
        if policy == "replace":
            pts["vis"] = np.random.default_rng(p).integers(0, 3, n).astype(np.uint8)
        rgb = torch.empty((3, n), dtype=torch.float32, device="cuda")
        gpu.eval_batch(P.points_to_device(pts), rgb)
        gpu.sync()
        ref.run_batch(pts)
        g, r = gpu.stats(), ref.stats()
        for k in ("lookups", "hits", "candidates", "inserted", "dropped_dup", "dropped_full", "replaced"):
            assert g[k] == r[k], (p, k)
    assert np.array_equal(gpu.table()[0], ref.table()[0])
