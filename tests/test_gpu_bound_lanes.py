"""The bound and calibration-target kernels by lane groups (csrc/bound.cu): the same
tiles in a call small enough to give each arm and sign its own lane, in a call large
enough for one lane an arm, and on the plain path (one thread a tile, FP64
throughout), for every number of arms, odd tile counts, point tiles and wide boxes."""
import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DESIGNS = {1: W.ONE_ARM, 2: W.TWO_ARM, 4: W.Design("berry4_n12", "berry4", 4, (12,), arm_null=W.BERRY4.arm_null)}


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _run(B, ctx, tiles, n):
    dt = B.DeviceTiles(tiles)
    lam = {1: -1.2, 2: -1.2, 4: 0.4}[tiles.d]
    s = ctx.step(dt, lam, 0.02, 0.05)
    lo = ctx.validate_lower(dt, lam, 0.02)
    cal = ctx.calibrate(dt, 0.05)
    torch.cuda.synchronize()
    ctx.sync()
    out = dict(u0=s["u0"], bound=s["bound"], alpha_prime=s["alpha_prime"], alpha_cal=cal["alpha_prime"],
               l0=lo["l0"], lower=lo["lower"])
    return {k: v[:n].cpu().numpy() for k, v in out.items()}


@pytest.mark.parametrize("d", [1, 2, 4])
def test_lane_groups_agree(B, d):
    rng = np.random.default_rng(d)
    n, big = 37, {1: 30001, 2: 16001, 4: 8001}[d]
    h = np.exp(rng.uniform(np.log(1e-4), np.log(1.0), (big, d)))
    h[:6] = 0.0                                     # a point: alpha' = alpha, bound = u0
    h[6] = 3.0
    tiles = W.from_centers(rng.uniform(-3.0, 1.0, (big, d)).round(2), h, 1, rng.integers(1, 3000, big).astype(np.int32))
    ctx = B.Context(DESIGNS[d], seed=2, K_max=3000)
    assert n * 2 * d < 152 * 4 * 32 * 3 < big * 2 * d     # one launch on each side of the rule
    few, many = _run(B, ctx, tiles.subset(np.arange(n)), n), _run(B, ctx, tiles, n)
    ctx.set_option(B.OPT_PLAIN, 1)
    plain = _run(B, ctx, tiles.subset(np.arange(n)), n)
    for k in few:
        assert np.allclose(few[k], many[k], rtol=1e-12, atol=1e-15), k
        # 1 - U loses its digits where U is near 1: absolute there
        assert np.allclose(few[k], plain[k], rtol=1e-12, atol=1e-12 if k == "lower" else 1e-15), k
    assert np.allclose(few["alpha_prime"][:6], 0.05, rtol=1e-14)
