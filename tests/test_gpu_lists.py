"""Insert through per-cell lists against the binned insert and the oracle: the same table,
counters and outputs.  N_e that are and are not multiples of four, cell counts that are no power
of two, cells with more keys than room (a skewed batch, one entry per cell), and a single
cell with thousands of candidates."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu

STATS = ("lookups", "hits", "candidates", "inserted", "dropped_dup", "dropped_full")


def _run(cache, pts):
    import torch
    n = len(pts["u"])
    rgb = torch.empty((3, n), dtype=torch.float32, device="cuda")
    hits = torch.empty(n, dtype=torch.int16, device="cuda")
    cache.eval_batch(P.points_to_device(pts), rgb, hits)
    cache.sync()
    return rgb.cpu().numpy(), hits.cpu().numpy()


def _points(kind, n, seed, n_mats):
    pts = W.points_uniform(n, seed=seed, n_mats=n_mats)
    if kind == "skewed":      # half of the points in 64 texels of one network
        k = np.arange(n) % 2 == 0
        pts["mat"][k] = 0
        pts["u"][k] = np.floor(pts["u"][k] * 8) / 1024
        pts["v"][k] = np.floor(pts["v"][k] * 8) / 1024
    if kind == "one texel":
        pts["mat"][:] = 0
        pts["u"][:], pts["v"][:] = 0.25, 0.75
    return pts


@pytest.mark.parametrize("kind,n_cells,entries", [("uniform", 1 << 16, 8), ("uniform", 70001, 4), ("uniform", 65537, 5),
                                                  ("uniform", 99991, 1), ("skewed", 1 << 17, 8), ("skewed", 66000, 7),
                                                  ("one texel", 1 << 16, 8)])
def test_lists_equal_bins(kind, n_cells, entries):
    mats = W.random_materials(8, 60, 120, 0.3, seed=9)
    roots = sum(len(P.analyze_material(m)["roots"]) for m in mats) / len(mats)
    n = int(300_000 / roots) + 77
    lists = P.Cache(mats, n_cells, entries)
    other = P.Cache(mats, n_cells, entries, flags=P.PMC_INSERT_BINNED)
    for p in range(2):
        pts = _points(kind, n, p, len(mats))
        a, b = _run(lists, pts), _run(other, pts)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        sa, sb = lists.stats(), other.stats()
        assert all(sa[k] == sb[k] for k in STATS), {k: (sa[k], sb[k]) for k in STATS}
        ta, tb = lists.table(), other.table()
        assert np.array_equal(ta[0], tb[0]) and np.array_equal(ta[1], tb[1])
    assert sa["inserted"] > 0 and (kind != "one texel" or sa["dropped_dup"] > 3072)


def test_lists_match_oracle():
    mats = W.random_materials(8, 60, 120, 0.3, seed=9)
    roots = sum(len(P.analyze_material(m)["roots"]) for m in mats) / len(mats)
    n = int(300_000 / roots)
    gpu, ref = P.Cache(mats, 1 << 16, 8), O.Cache(mats, 1 << 16, 8, level=10, threads=16)
    pts = _points("skewed", n, 3, len(mats))
    rgb, hits = _run(gpu, pts)
    r = ref.run_batch(pts)
    assert np.abs(rgb - r["rgb"]).max() <= 1e-4
    g, s = gpu.stats(), ref.stats()
    assert all(g[k] == s[k] for k in STATS)
    assert np.array_equal(gpu.table()[0], ref.table()[0])
