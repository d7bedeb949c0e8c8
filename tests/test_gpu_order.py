"""Work items in descending cost of their networks, and one or two points per lane by the size of
the batch: networks of very uneven and of equal length, at a single point, at a warp's edges,
and at batches on both sides of the line, against the oracle; the large batches also bit for bit
against one point per lane throughout."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu

TOL = 1e-4   # the FP32 path's tolerance against FP64


def _mats(kind):
    if kind == "uneven":   # the longest neither first nor last
        small = W.random_materials(12, 5, 12, 0.3, seed=3)
        return small[:7] + W.random_materials(1, 300, 300, 0.3, seed=4) + small[7:]
    return W.random_materials(1, 10, 10, 0.3, seed=5) * 3


def _run(mats, pts, cells, schedule):
    import torch
    c = P.Cache(mats, cells or 1, 8, flags=0 if cells else P.PMC_CACHE_OFF)
    c.set_schedule(schedule)
    n = len(pts["u"])
    d, out = P.points_to_device(pts), []
    for _ in range(2):
        rgb = torch.full((3, n), 7.0, device="cuda")
        hits = torch.full((n,), 99, dtype=torch.int16, device="cuda")
        c.eval_batch(d, rgb, hits)
        c.sync()
        out.append((rgb.cpu().numpy(), hits.cpu().numpy().astype(np.uint16)))
    return out, c.stats()


@pytest.mark.parametrize("cells", [0, 4096])
@pytest.mark.parametrize("kind", ["uneven", "equal"])
@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_small_batches_match_oracle(kind, n, cells):
    mats = _mats(kind)
    pts = W.points_uniform(n, seed=n, n_mats=len(mats))
    pts["u"] = np.round(pts["u"] * 16) / 16
    pts["v"] = np.round(pts["v"] * 16) / 16
    ref = O.Cache(mats, cells, 8, level=10, cache_off=not cells)
    out, st = _run(mats, pts, cells, 0)
    for rgb, hits in out:
        r = ref.run_batch(pts)
        assert np.abs(rgb - r["rgb"]).max() <= TOL and np.array_equal(hits, r["hits"])
    assert all(st[k] == ref.stats()[k] for k in ("lookups", "hits", "inserted"))


@pytest.mark.parametrize("cells", [0, 1 << 16])
@pytest.mark.parametrize("kind,n", [("equal", 100_003), ("equal", 200_001), ("uneven", 900_001)])
def test_large_batches_match_one_point(kind, n, cells):
    mats = _mats(kind)
    pts = W.points_uniform(n, seed=n, n_mats=len(mats))
    (a, sa), (b, sb) = (_run(mats, pts, cells, f) for f in (0, P.PMC_ONE_POINT))
    for (r0, h0), (r1, h1) in zip(a, b):
        assert np.array_equal(r0, r1) and np.array_equal(h0, h1)
    assert sa == sb


@pytest.mark.parametrize("n", [60_000, 150_001, 400_003])
@pytest.mark.parametrize("kind", ["equal", "wide"])
def test_batched_misses_match_one_point(kind, n):
    """Second and third passes whose misses fill fewer or more items than the line for two misses
    per lane, and a program whose values fill more than its row file's limit."""
    if kind == "wide":
        b = W.Builder()
        uv = b.add(W.OP_UV)
        v = [b.add(W.OP_FBM, [uv], ip=[1, k], fp=[1.0 + 0.05 * k, 2.0, 0.5]) for k in range(60)]
        r = v[0]
        for x in v[1:] + v[::-1]:
            r = b.add(W.OP_MIX, [r, x], fp=[0.3])
        b.add(W.OP_MUL, [r, b.add(W.OP_FACING, [b.add(W.OP_NORMAL)], fp=[0.2, 0.5, 0.4])])
        mats = [b.build()]
    else:
        mats = W.random_materials(2, 10, 10, 0.3, seed=5)
    passes = [W.points_uniform(n, seed=s, n_mats=len(mats)) for s in (1, 2, 3)]
    res = []
    import torch
    for flags in (0, P.PMC_ONE_POINT):
        c = P.Cache(mats, 1 << 16, 8)
        c.set_schedule(flags)
        out = []
        for p in passes:
            rgb, hits = torch.empty((3, n), device="cuda"), torch.empty(n, dtype=torch.int16, device="cuda")
            c.eval_batch(P.points_to_device(p), rgb, hits)
            c.sync()
            out += [rgb.cpu().numpy(), hits.cpu().numpy()]
        assert out[3].any() and c.stats()["misses"] > n
        res.append(out + [c.stats()["inserted"], c.stats()["nodes_evaluated"]] + list(c.table()))
    for x, y in zip(*res):
        assert np.array_equal(x, y)
