"""The basket simulation evaluates only the trials that a bit per count state does
not rule out (csrc/sim_basket.cu).  Its outputs are exact, so they are compared bit
for bit with the direct mode, which evaluates every trial with the same posterior
function and selects with its own radix passes: every null mask (none included),
windows that hold every count and windows cut off at their largest width, centres
far out (counts at 0 and n only), K at the edges of the sample, the sixteen-trial
words and the steps, and thresholds from "nothing rejects" to "everything does"."""
import math

import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EDGES = (1, 2, 15, 16, 17, 511, 513, 2047, 2048, 2049, 2064, 4097, 4607, 4608, 4609, 8705, 13001)


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _tiles(n, K, seed):
    rng = np.random.default_rng(seed)
    ax = np.concatenate([np.linspace(-3.5, 1.0, 21), [-9.0, 9.0]])
    c = ax[rng.integers(0, ax.size, (n, 4))]
    mask = rng.integers(1, 16, n).astype(np.uint32)
    mask[0] = 16                                    # none of the four arms: S = +inf
    return W.from_centers(c, 0.02, mask, np.asarray(K)[rng.integers(0, len(K), n)].astype(np.int32))


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


@pytest.mark.parametrize("n,n_tiles", [(1, 40), (7, 60), (19, 60), (20, 60), (35, 700), (63, 60)])
def test_candidates_match_every_trial(B, n, n_tiles):
    design = W.Design("berry4", "berry4", 4, (n,), arm_null=W.BERRY4.arm_null)
    tiles = _tiles(n_tiles, EDGES, 7)
    ctx = B.Context(design, seed=3, K_max=int(tiles.K.max()))
    dt = B.DeviceTiles(tiles)
    lams = (0.0, 0.15, 1e-4, 0.6, 1.0, math.inf)
    a = _outputs(ctx, dt, lams, (0.025, 0.6))
    ctx.set_option(B.OPT_BAYES_DIRECT, 1)
    b = _outputs(ctx, dt, lams, (0.025, 0.6))
    for j, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y), j


def test_candidates_beyond_a_block_of_steps(B):
    """K past the 64 steps of 2,048 trials that a queue entry can address."""
    K = np.array([131072 + 511, 131072 + 512, 131072 + 513, 133120 + 512, 262144 + 513, 300001])
    tiles = W.from_centers(np.linspace(-2.5, 0.8, 24).reshape(6, 4), 0.02, np.array([15, 1, 6, 9, 3, 12], np.uint32),
                           K.astype(np.int32))
    ctx = B.Context(W.BERRY4, seed=9, K_max=int(K.max()))
    dt = B.DeviceTiles(tiles)
    a = _outputs(ctx, dt, (0.0, 0.15), (0.025,))
    ctx.set_option(B.OPT_BAYES_DIRECT, 1)
    b = _outputs(ctx, dt, (0.0, 0.15), (0.025,))
    for j, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y), j
