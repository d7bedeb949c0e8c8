"""Binned insert with bins of fewer than 256 cells (many candidates for the table's size):
tables whose cell count is no multiple of the bin, down to a single cell, against the
oracle's sequential insert."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells,entries,flags", [(1, 8, "binned"), (33, 8, "binned"), (300, 8, "replace"),
                                                   (129, 16, "keep"), (1000, 8, "replace"), (8191, 8, "binned")])
def test_small_bins_match_oracle(n_cells, entries, flags):
    import torch
    mats = W.random_materials(6, 40, 90, 0.3, seed=5)
    roots = max(len(P.analyze_material(m)["roots"]) for m in mats)
    n = 12001
    assert n_cells > 300 or n * roots > 1024 * max(1, n_cells // 256)   # bins shrink
    gpu = P.Cache(mats, n_cells, entries, flags={"binned": P.PMC_INSERT_BINNED, "replace": P.PMC_REPLACE_VISIBILITY,
                                                  "keep": 0}[flags])
    ref = O.Cache(mats, n_cells, entries, level=10, replacement=flags == "replace")
    for p in range(2):
        pts = W.points_uniform(n, seed=p, n_mats=len(mats))
        if flags == "replace":
            pts["vis"] = np.random.default_rng(p).integers(0, 3, n).astype(np.uint8)
        rgb = torch.empty((3, n), dtype=torch.float32, device="cuda")
        gpu.eval_batch(P.points_to_device(pts), rgb)
        gpu.sync()
        ref.run_batch(pts)
    g, r = gpu.stats(), ref.stats()
    for k in ("lookups", "hits", "candidates", "inserted", "dropped_dup", "dropped_full", "replaced"):
        assert g[k] == r[k], k
    assert np.array_equal(gpu.table()[0], ref.table()[0])
