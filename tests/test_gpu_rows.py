"""Value rows of the interpreter on the GPU: nodes whose three channels are equal keep one row
(noise, Worley, facing and arithmetic on them), and every operator reads one-row and
three-row inputs alike; noise and Worley at arguments on both sides of the limit of the fast
floor.  Against the FP64 oracle, with one and two points per lane."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_07238_gb300 import pmc as P
from paper_2305_07238_gb300 import workload as W

pytestmark = pytest.mark.gpu

TOL = 1e-4   # the FP32 path's tolerance against FP64


def _sources(b):
    """A one-row value, a three-row value, and constants of either kind."""
    uv = b.add(W.OP_UV)
    noise = b.add(W.OP_FBM, [uv], ip=[2, 5], fp=[4.0, 2.0, 0.5])
    ramp = b.add(W.OP_RAMP, [noise], ip=[2], fp=[0, 1, 0, 0, 0.1, 0.6, 0.3, 0.9, 0.2, 0.7])
    grey = b.add(W.OP_CONST, fp=[0.4, 0.4, 0.4])
    col = b.add(W.OP_CONST, fp=[0.9, 0.5, 0.3])
    wor = b.add(W.OP_VORONOI, [uv], ip=[0, 9], fp=[3.0])
    return {"m": noise, "w": wor, "c": ramp, "g": grey, "k": col, "uv": uv}


def _binary(op, x, y):
    b = W.Builder()
    s = _sources(b)
    r = b.add(op, [s[x], s[y]], fp=[0.3] if op == W.OP_MIX else [])
    b.add(W.OP_ADD, [r, b.add(W.OP_FACING, [b.add(W.OP_NORMAL)], fp=[0.1, 0.2, 0.1])])
    return b.build()


def _unary(op, x, fp, ip=()):
    b = W.Builder()
    s = _sources(b)
    r = b.add(op, [s[x]], fp=fp, ip=ip)
    b.add(W.OP_MUL, [r, s["k"]])
    return b.build()


def _mono_output():
    """The material output itself has equal channels."""
    b = W.Builder()
    s = _sources(b)
    b.add(W.OP_MUL, [s["m"], b.add(W.OP_FACING, [b.add(W.OP_NORMAL)], fp=[0.6, 0.0, 0.8])])
    return b.build()


NETS = ([_binary(op, x, y) for op in (W.OP_ADD, W.OP_MUL, W.OP_MIX)
         for x, y in (("m", "w"), ("m", "c"), ("c", "m"), ("c", "k"), ("g", "m"), ("k", "w"), ("g", "g"))]
        + [_unary(W.OP_POW, x, [1.7]) for x in ("m", "c")]
        + [_unary(W.OP_FACING, x, [0.3, 0.5, 0.2]) for x in ("m", "c", "uv")]
        + [_unary(W.OP_FBM, "m", [3.0, 2.0, 0.5], [2, 1]), _unary(W.OP_VORONOI, "m", [3.0], [0, 4]), _mono_output()])


@pytest.mark.parametrize("flags", [0, P.PMC_ONE_POINT, P.PMC_UNSORTED])
@pytest.mark.parametrize("off", [False, True])
def test_every_operator_reads_either_kind_of_row(flags, off):
    import torch
    n = 4001
    gpu = P.Cache(NETS, 4096, 8, flags=flags | (P.PMC_CACHE_OFF if off else 0))
    ref = O.Cache(NETS, 4096, 8, level=10, cache_off=off)
    for p in range(2):
        pts = W.points_uniform(n, seed=p, n_mats=len(NETS))
        pts["u"][::2] = np.round(pts["u"][::2] * 16) / 16      # shared texels: hits in the second pass
        pts["v"][::2] = np.round(pts["v"][::2] * 16) / 16
        rgb = torch.empty((3, n), dtype=torch.float32, device="cuda")
        hits = torch.empty(n, dtype=torch.int16, device="cuda")
        gpu.eval_batch(P.points_to_device(pts), rgb, hits)
        gpu.sync()
        r = ref.run_batch(pts)
        assert np.abs(rgb.cpu().numpy() - r["rgb"]).max() <= TOL
        assert np.array_equal(hits.cpu().numpy().astype(np.uint16), r["hits"])


@pytest.mark.parametrize("flags", [0, P.PMC_ONE_POINT])
@pytest.mark.parametrize("op", [W.OP_FBM, W.OP_VORONOI])
def test_noise_on_both_sides_of_the_fast_floor(op, flags):
    """Coordinates around and beyond 2^22, exact in FP32 with a scale of 1, so that FP32 and
    FP64 see the same argument; odd lanes stay small, so that both forms run in one warp."""
    import torch
    b = W.Builder()
    b.add(op, [b.add(W.OP_POSITION)], ip=[1, 7], fp=[1.0, 2.0, 0.5])
    mat = b.build()
    n = 2048
    pts = W.points_uniform(n, seed=3)
    rng = np.random.default_rng(4)
    for k in ("px", "py"):
        big = np.ldexp(1.0, rng.integers(20, 25, n)) * rng.choice([-1.0, 1.0], n) + rng.integers(-8, 8, n) * 0.25
        pts[k] = np.where(np.arange(n) % 2 == 0, big, rng.integers(-4000, 4000, n) / 64.0).astype(np.float32)
    pts["px"][:4] = [2.0**22, -(2.0**22), 2.0**22 - 0.5, -(2.0**22) - 0.5]
    gpu = P.Cache([mat], 64, 8, flags=flags | P.PMC_CACHE_OFF)
    rgb = torch.empty((3, n), dtype=torch.float32, device="cuda")
    gpu.eval_batch(P.points_to_device(pts), rgb)
    gpu.sync()
    ref = O.Cache([mat], 64, 8, level=10, cache_off=True).run_batch(pts)
    assert np.abs(rgb.cpu().numpy() - ref["rgb"]).max() <= TOL
