"""The four-arm simulation kernel evaluates only the trials whose final counts can
give a small statistic (csrc/sim_bayes4.cu).  Its outputs are exact, so they are
compared bit for bit with the direct mode, which evaluates every trial with the
same posterior function and selects with its own radix passes: every design form
(packed with scores, packed with raw counts, byte form), both tile groupings,
every mask (none counted included), K at the edges of the sample, the sixteen-trial
words and the steps, and thresholds from "nothing rejects" to "everything does"."""
import math

import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EDGES = (1, 2, 15, 16, 17, 511, 512, 513, 1023, 1024, 1025, 1040, 2559, 2560, 2561, 2577, 4607, 4609, 18001)


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _tiles(n, K, seed, lo=-3.0, hi=3.0):
    rng = np.random.default_rng(seed)
    ax = np.linspace(lo, hi, 23)
    c = ax[rng.integers(0, ax.size, (n, 4))]
    near = rng.random(n) < 0.5                      # half the tiles near the null boundary
    c[near] = c[near][:, :1] + 0.25 * rng.integers(-1, 2, (int(near.sum()), 4))
    mask = rng.integers(1, 16, n).astype(np.uint32)
    mask[:8] = np.arange(1, 9)[:n]                  # 8: no treatment counted, S = +inf
    Ka = np.asarray(K)[rng.integers(0, len(K), n)] if np.ndim(K) else np.full(n, K)
    return W.from_centers(c, 0.02, mask, Ka.astype(np.int32))


def _outputs(ctx, dt, lams, alphas):
    out = []
    for lam in lams:
        out += [x.clone() for x in ctx.simulate_tiles(dt, lam)]
    for alpha in alphas:
        s = ctx.step(dt, lams[1], 0.01, alpha)
        out += [s[k].clone() for k in ("R", "Xrej", "score", "lambda_tile", "lam")]
        cal = ctx.calibrate(dt, alpha)
        out += [cal["lambda_tile"].clone(), torch.tensor(cal["lam"])]
    torch.cuda.synchronize()
    ctx.sync()
    return out


@pytest.mark.parametrize("looks", [(10, 20, 40), (15, 30, 60), (2, 5, 115), (20, 40, 70), (3, 4, 128)])
@pytest.mark.parametrize("n_tiles", [40, 2432])
def test_candidates_match_every_trial(B, looks, n_tiles):
    design = W.Design("bayes4", "bayes4", 4, looks)
    tiles = _tiles(n_tiles, EDGES, 7)
    ctx = B.Context(design, seed=3, K_max=int(tiles.K.max()))
    dt = B.DeviceTiles(tiles)
    lams = (0.0, 0.06, 1e-5, 0.6, 1.0, math.inf)
    a = _outputs(ctx, dt, lams, (0.025, 0.6))
    ctx.set_option(B.OPT_BAYES_DIRECT, 1)
    b = _outputs(ctx, dt, lams, (0.025, 0.6))
    for j, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y), j


def test_candidates_at_large_K_and_offsets(B):
    """K = 2^20 with a count table beyond 4 GB (64-bit row offsets), against the same
    tiles on a table that holds only their own axis values."""
    K = 1 << 20
    few = _tiles(6, K, 11, -1.0, 1.0).with_K([K, K - 1, 70000, 66000, 65536, 3])
    wide = W.TileSet(4, [np.concatenate([a, np.linspace(4.0, 5.0, 515)]) for a in few.axis], few.idx, few.halfwidth,
                     few.null_mask, few.K)
    assert 2 * sum(len(a) for a in wide.axis) * K > 1 << 32
    ctx = B.Context(W.BAYES4, seed=5, K_max=K)
    a = _outputs(ctx, B.DeviceTiles(few), (0.0, 0.06), (0.025,))
    b = _outputs(ctx, B.DeviceTiles(wide), (0.0, 0.06), (0.025,))
    for j, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y), j
