"""Training kernel: masters and moments kept in registers over a launch are the ones in memory
between launches, so any split of the steps over launches gives the same bits."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2305_07238_gb300 import pmc as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", [(1,) * 7, (3, 4), (6, 1)])
def test_steps_over_launches_equal_steps_in_one(parts):
    import torch
    rng = np.random.default_rng(11)
    n = 512
    data = torch.from_numpy(rng.random((n, 5)).astype(np.float32)).cuda()
    th0 = torch.from_numpy(rng.normal(0.0, 0.2, M.N_PARAMS).astype(np.float32))

    def train(launches):
        theta, m, v = th0.cuda(), torch.zeros(M.N_PARAMS, device="cuda"), torch.zeros(M.N_PARAMS, device="cuda")
        done = 0
        for k in launches:
            P.mlp_train(theta, m, v, data, k, done, 7, 1e-2)
            done += k
        return torch.stack([theta, m, v]).cpu()

    whole = train((7,))
    assert not torch.equal(whole[0], th0)
    assert torch.equal(train(parts), whole)
