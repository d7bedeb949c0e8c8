"""Materials out of range are counted and reported, whichever launches group the batch: one cluster, the
last block of the histogram, or a launch of its own; a batch without any raises nothing."""
import numpy as np
import pytest

from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 8192, 8193])
@pytest.mark.parametrize("n_mats", [1, 1024, 1025])
@pytest.mark.parametrize("share", [0.0, 0.05, 1.0])
def test_bad_materials_are_counted(n, n_mats, share):
    import torch
    c = P.Cache([W.material_tiny()] * n_mats, 4096, 8)
    pts = W.points_uniform(n, seed=n, n_mats=n_mats)
    rng = np.random.default_rng(n)
    bad = rng.random(n) < share
    pts["mat"] = np.where(bad, n_mats + rng.integers(0, 3, n), pts["mat"]).astype(np.uint32)
    rgb = torch.full((3, n), 7.0, device="cuda")
    c.eval_batch(P.points_to_device(pts), rgb)
    if bad.any():
        with pytest.raises(P.PmcError) as e:
            c.sync()
        assert e.value.status == P.PMC_ERR_INVALID_ARG
    else:
        c.sync()
    s = c.stats()
    assert s["bad_points"] == bad.sum() and s["points"] == n and s["lookups"] == n - bad.sum()
    assert not rgb.cpu().numpy()[:, bad].any()
