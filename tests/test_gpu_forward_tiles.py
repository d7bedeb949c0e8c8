"""Stand-alone surrogate network at the edges of its 128-row tiles and of its persistent grid,
against the oracle's network with the same BF16 rounding points."""
import numpy as np
import pytest

from oracle import mlp as M
from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P

pytestmark = pytest.mark.gpu

MAX, Q99 = 2e-2, 1e-4   # the forward pass's tolerance: a flipped BF16 rounding, and the rest


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 760 * 128 - 1, 760 * 128 + 1, 2 * 760 * 128 + 65])
def test_forward_at_tile_edges(n):
    import torch
    rng = np.random.default_rng(n)
    th = M.bf16_round(rng.normal(0.0, 0.25, M.N_PARAMS))
    u, v = rng.random(n).astype(np.float32), rng.random(n).astype(np.float32)
    out = P.mlp_forward(torch.as_tensor(th, dtype=torch.float32).cuda(), torch.from_numpy(u).cuda(),
                        torch.from_numpy(v).cuda(), clamp=False).cpu().numpy()
    k = np.unique(np.concatenate([np.arange(min(n, 300)), np.arange(max(0, n - 300), n)]))   # first and last rows
    ref = O.mlp_forward(th, u[k].astype(np.float64), v[k].astype(np.float64), bf16=True).T
    err = np.abs(out[:, k] - ref)
    assert np.isfinite(out).all() and err.max() <= MAX and np.quantile(err, 0.99) <= Q99
