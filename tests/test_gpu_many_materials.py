"""Layout of the materials' segments and work items around the number of materials from which two
blocks of a launch of their own do it: with surrogates, and with more probes than the scratch holds."""
import numpy as np
import pytest

from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _batch(pts):
    import torch
    n = len(pts["mat"])
    return P.points_to_device(pts), torch.empty((3, n), device="cuda"), torch.empty(n, dtype=torch.int16, device="cuda")


@pytest.mark.parametrize("n_mats", [1024, 1025, 9001])
def test_surrogates_of_many_materials(n_mats):
    # copies of one network, every hundredth with a surrogate, against two copies of it
    net = W.surrogate_materials(1, 60, 90, seed=3)[0]
    theta = np.random.default_rng(1).normal(0.0, 0.2, P.MLP_PARAMS).astype(np.float32)
    pts = W.points_uniform(30001, seed=4, n_mats=n_mats)
    out = []
    for many in (True, False):
        c = P.Cache([net] * (n_mats if many else 2), 1 << 15, 8)
        for m in range(0, n_mats, 100) if many else [0]:
            c.set_surrogate(m, theta)
        p = dict(pts) if many else {**pts, "mat": (pts["mat"] % 100 != 0).astype(np.uint32)}
        d, rgb, hits = _batch(p)
        c.eval_batch(d, rgb, hits)
        c.sync()
        out.append((rgb.cpu().numpy(), {k: c.stats()[k] for k in ("surrogate_evals", "lookups", "points", "nodes_evaluated")}))
    assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    assert 0 < out[0][1]["surrogate_evals"] < 30001


@pytest.mark.parametrize("n_mats", [1024, 1025, 9001])
def test_too_many_probes_for_the_scratch(n_mats):
    net = W.material_tiny()
    n = 20000
    pts = W.points_uniform(n, seed=2, n_mats=n_mats)
    c = P.Cache([net] * n_mats, 4096, 8, probe_capacity=n - 1)
    d, rgb, hits = _batch(pts)
    c.eval_batch(d, rgb, hits)
    with pytest.raises(P.PmcError) as e:
        c.sync()
    assert e.value.status == P.PMC_ERR_UNSUPPORTED
    s = c.stats(check=False)
    assert s["nodes_evaluated"] == s["inserted"] == 0
    c.reset()
    d, rgb, hits = _batch({k: v[: n - 1] for k, v in pts.items()})
    c.eval_batch(d, rgb, hits)
    c.sync()
    assert c.stats()["lookups"] == n - 1
