"""The scans run by the last block of the grouping and lookup kernels: material counts around the
block's threads and beyond the shared-memory histogram, cacheable nodes on both sides of
the lookup's limit (2048), and an empty batch."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _small(rng):
    """A network with one cacheable node, varied by its seed."""
    b = W.Builder()
    n = b.add(W.OP_FBM, [b.add(W.OP_UV)], ip=[1, int(rng.integers(1 << 20))], fp=[3.0, 2.0, 0.5])
    r = b.add(W.OP_POW, [n], fp=[1.5])
    b.add(W.OP_MUL, [r, b.add(W.OP_FACING, [b.add(W.OP_NORMAL)], fp=[0.2, 0.5, 0.4])])
    return b.build()


@pytest.mark.parametrize("n_mats", [1, 255, 257, 1025, 2047, 2049, 4099])
def test_scans_match_oracle(n_mats):
    import torch
    rng = np.random.default_rng(n_mats)
    mats = [_small(rng) for _ in range(n_mats)]
    gpu, ref = P.Cache(mats, 4096, 8), O.Cache(mats, 4096, 8, level=10)
    for p, n in enumerate((9001, 0, 9001)):
        pts = W.points_uniform(max(n, 1), seed=1 + p // 2, n_mats=n_mats)
        pts = {k: v[:n] for k, v in pts.items()}
        pts["u"] = np.round(pts["u"] * 8) / 8
        rgb = torch.empty((3, n), dtype=torch.float32, device="cuda")
        hits = torch.empty(n, dtype=torch.int16, device="cuda")
        gpu.eval_batch(P.points_to_device(pts), rgb, hits)
        gpu.sync()
        if n:
            r = ref.run_batch(pts)
            assert np.abs(rgb.cpu().numpy() - r["rgb"]).max() <= 1e-4
            assert np.array_equal(hits.cpu().numpy().astype(np.uint16), r["hits"])
    g, r = gpu.stats(), ref.stats()
    for k in ("lookups", "hits", "inserted"):
        assert g[k] == r[k], k
    assert g["batches"] == 3 and g["points"] == 2 * 9001
