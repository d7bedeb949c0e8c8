"""Training kernel: masters and moments kept in registers over a launch are the ones in memory
between launches, so any split of the steps over launches gives the same bits; and a whole
training call, whose pairs are drawn in parts beside the training."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

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


_M64 = (1 << 64) - 1


def _mix(z):
    """SplitMix64's output function of the states z (uint64)."""
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _initial(seed):
    """He-uniform weights, zero biases, output bias 1/2."""
    k = np.arange(1, 4096 * 2 + 192 + 1, dtype=np.uint64)
    r = (_mix(np.uint64(seed & _M64) + k * np.uint64(0x9E3779B97F4A7C15)) >> np.uint64(11)) / 2.0**53
    lim = np.sqrt(6.0 / 64.0)
    th = np.zeros(M.N_PARAMS, np.float32)
    th[:4096] = (2.0 * r[:4096] - 1.0) * lim
    th[4160:8256] = (2.0 * r[4096:8192] - 1.0) * lim
    th[8320:8512] = (2.0 * r[8192:] - 1.0) * lim * 0.5
    th[8512:] = 0.5
    return th


def _pairs(net, seed, mi, n):
    """The pairs of network mi: (u, v) from the generator, the value from an uncached pass."""
    import torch
    row = np.arange(n, dtype=np.uint64) | np.uint64(mi << 32)
    x = _mix((np.uint64(seed) ^ row) + np.uint64(0x9E3779B97F4A7C15))
    pts = {"mat": np.zeros(n, np.uint32)}
    pts["u"] = ((x >> np.uint64(40)).astype(np.float32) / np.float32(1 << 24)).astype(np.float32)
    pts["v"] = (((x >> np.uint64(8)) & np.uint64(0xFFFFFF)).astype(np.float32) / np.float32(1 << 24)).astype(np.float32)
    for k in ("px", "py", "pz", "nx", "ny", "nz"):
        pts[k] = np.zeros(n, np.float32)
    rgb = torch.empty((3, n), device="cuda")
    c = P.Cache([net], 1, 8, flags=P.PMC_CACHE_OFF)
    c.eval_batch(P.points_to_device(pts), rgb)
    c.sync()
    uv = torch.from_numpy(np.stack([pts["u"], pts["v"]])).cuda()
    return torch.cat([uv, rgb]).T.contiguous()


def _net(layers, seed):
    """A network whose output is its cacheable node."""
    b = W.Builder()
    r = b.add(W.OP_FBM, [b.add(W.OP_UV)], ip=[2, seed], fp=[1.0, 2.0, 0.5])
    for k in range(layers):
        f = b.add(W.OP_FBM, [b.add(W.OP_UV)], ip=[1 + k % 3, seed + k], fp=[1.0 + 0.3 * k, 2.0, 0.5])
        c = b.add(W.OP_CONST, fp=[0.9, 0.5, 0.2])
        r = b.add(W.OP_MIX, [r, b.add(W.OP_MUL, [f, c])], fp=[0.4])
    return b.build()


def _wide(n):
    """A network that holds n values at a time."""
    b = W.Builder()
    uv = b.add(W.OP_UV)
    v = [b.add(W.OP_FBM, [uv], ip=[1, k], fp=[1.0 + 0.05 * k, 2.0, 0.5]) for k in range(n)]
    r = v[0]
    for x in v[1:] + v[::-1]:
        r = b.add(W.OP_MIX, [r, x], fp=[0.3])
    return b.build()


@pytest.mark.parametrize("wide", [2, 100])   # two points per lane, one
@pytest.mark.parametrize("n_train,n_valid,epochs", [(128, 1, 1), (4096, 1000, 2), (8192, 1000, 2), (32768, 4099, 1)])
def test_training_beside_the_drawing_of_its_pairs(n_train, n_valid, epochs, wide):
    """The call draws its pairs in parts (none below 64 steps an epoch, two, eight) while it
    trains; the result has the bits of training on the whole set of pairs."""
    import torch
    nets = [_net(2, 5), _net(9, 6), _wide(wide), _net(4, 7)]
    c = P.Cache(nets, 64, 8)
    seed = 21
    rmse = c.train_surrogates(n_train=n_train, n_valid=n_valid, epochs=epochs, lr=1e-2, seed=seed)
    again = c.train_surrogates(n_train=n_train, n_valid=n_valid, epochs=epochs, lr=1e-2, seed=seed)
    assert np.array_equal(rmse, again)
    steps = n_train // 128 * epochs
    for m, net in enumerate(nets):
        got = c.get_surrogate(m)
        assert got["node"] == len(net) - 1
        theta = torch.from_numpy(_initial(seed * 0x100000001B3 + m + 1)).cuda()
        m1, m2 = torch.zeros_like(theta), torch.zeros_like(theta)
        P.mlp_train(theta, m1, m2, _pairs(net, seed, m, n_train), steps, 0, steps, 1e-2)
        assert np.array_equal(theta.cpu().numpy(), got["theta"])
        v = _pairs(net, seed ^ 0x5DEECE66D, m, n_valid)
        y = P.mlp_forward(theta, v[:, 0].contiguous(), v[:, 1].contiguous(), clamp=True)
        err = (y - v[:, 2:].T).double().square().mean().sqrt().item()
        assert rmse[m] == pytest.approx(err, rel=1e-5)
