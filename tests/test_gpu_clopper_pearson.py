"""The Clopper-Pearson solve by groups of lanes (csrc/bound.cu) against the oracle:
R from 0 to K, K at the edges of its branches (the small-R sum, the continued
fraction, few trials), confidence levels on both sides of one half, and the two
group widths (few keys and more than 40,000 distinct keys)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu

RTOL = 1e-12   # the bar of every FP64 bound of this library


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _tiles(n, K_hi, seed, K_lo=1):
    rng = np.random.default_rng(seed)
    c = rng.uniform(-1.5, 3.0, (n, 1))
    K = np.exp(rng.uniform(np.log(K_lo), np.log(K_hi), n)).astype(np.int32)
    K[:16] = [1, 2, 9, 10, 11, 39, 40, 41, 49, 50, 51, 80, 81, 82, K_hi - 1, K_hi]
    return W.from_centers(c, 0.01, np.ones(n, np.uint32), K)


@pytest.mark.parametrize("delta", [0.01, 0.2, 0.5, 0.7, 1e-6])
def test_upper_and_lower_against_the_oracle(B, delta):
    tiles = _tiles(700, 60000, 3)
    ctx = B.Context(W.ONE_ARM, seed=9, K_max=60000)
    dt = B.DeviceTiles(tiles)
    up, lo = ctx.validate(dt, -1.96, delta), ctx.validate_lower(dt, -1.96, delta)
    torch.cuda.synchronize()
    ctx.sync()
    R = up["R"].cpu().numpy()
    assert (R == 0).any() and (R == tiles.K).any()
    ref_u = O.validate_bounds(W.ONE_ARM, tiles, R, delta)["u0"]
    ref_l = O.validate_lower(W.ONE_ARM, tiles, R, delta)["l0"]
    # R = K: P(Binom(K, l) >= K) = l^K = delta, so l = delta^(1/K); the oracle takes 1 - u there,
    # which keeps 1e-16 / delta of its digits for K = 1
    ref_l = np.where(R == tiles.K, np.exp(np.log(delta) / tiles.K), ref_l)
    assert np.allclose(up["u0"].cpu().numpy(), ref_u, rtol=RTOL, atol=0)
    assert np.allclose(lo["l0"].cpu().numpy(), ref_l, rtol=RTOL, atol=0)


def test_many_distinct_keys(B):
    tiles = _tiles(100000, 30000, 4, 3000)
    ctx = B.Context(W.ONE_ARM, seed=9, K_max=30000)
    out = ctx.validate(B.DeviceTiles(tiles), -1.96, 0.01)
    torch.cuda.synchronize()
    ctx.sync()
    R, u0 = out["R"].cpu().numpy(), out["u0"].cpu().numpy()
    assert len(np.unique(tiles.K.astype(np.int64) << 32 | R)) > 40000
    rows = np.random.default_rng(0).choice(tiles.n_tiles, 500, replace=False)
    rows[:16] = np.arange(16)
    ref = O.validate_bounds(W.ONE_ARM, tiles.subset(rows), R[rows], 0.01)["u0"]
    assert np.allclose(u0[rows], ref, rtol=RTOL, atol=0)
