"""The basket simulation at rates far from the null rates (csrc/sim_basket.cu), where S
lies near 0 or 1 throughout: the tiles whose sample shows this, and those whose order
statistic lies past their level, go to the kernel that evaluates every trial.  Whole
numbers and table values agree bit for bit with the direct form, at K around the sizes
where the form changes, in both block sizes, twice in a row on one context; and the
simulation takes no longer than it did with one gather for every trial."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _tiles(lo, hi, n_tiles, K, seed):
    rng = np.random.default_rng(seed)
    ax = np.linspace(lo, hi, 12)
    return W.TileSet(4, [ax] * 4, rng.integers(0, 12, (n_tiles, 4)).astype(np.int32), np.full((n_tiles, 4), 0.01),
                     rng.integers(1, 16, n_tiles).astype(np.uint32), K[rng.integers(0, len(K), n_tiles)].astype(np.int32))


def _outputs(ctx, dt):
    out = []
    for lam, alpha in ((0.15, 0.025), (0.15, 0.3), (1e-4, 0.1)):
        s = ctx.step(dt, lam, 0.01, alpha)
        out += [s[k].clone() for k in ("R", "Xrej", "lambda_tile", "lam")]
        c = ctx.calibrate(dt, alpha)
        out += [c["lambda_tile"].clone(), torch.tensor(c["lam"])]
    torch.cuda.synchronize()
    ctx.sync()
    return out


@pytest.mark.parametrize("n_tiles", [40, 900])
@pytest.mark.parametrize("n,lo,hi", [(35, 1.0, 4.0), (35, -6.0, -4.0), (35, -1.0, 2.0), (12, -2.0, 3.0), (63, -5.0, 3.0)])
def test_outputs_far_from_the_null_rates(B, n, lo, hi, n_tiles):
    tiles = _tiles(lo, hi, n_tiles, np.array([1, 511, 2048, 2049, 2560, 4000, 8192, 8193, 9001]), n)
    dt = B.DeviceTiles(tiles)
    ctx = B.Context(dataclasses.replace(W.BERRY4, looks=(n,)), seed=5, K_max=9001)
    a, again = _outputs(ctx, dt), _outputs(ctx, dt)
    ctx.set_option(B.OPT_BAYES_DIRECT, 1)
    for j, (x, y, z) in enumerate(zip(a, again, _outputs(ctx, dt))):
        assert torch.equal(x, y) and torch.equal(x, z), j


@pytest.mark.parametrize("lo,hi,us", [(1.0, 4.0, 366.0), (-6.0, -4.0, 409.0)])
def test_time_far_from_the_null_rates(B, lo, hi, us):
    """us: a step of the kernel that gathered for every trial, on this grid (8^4, K = 16,384)."""
    t = W.berry_grid(8, 16384)
    f = lambda a: (a + 3.5) / 4.5 * (hi - lo) + lo
    dt = B.DeviceTiles(W.TileSet(4, [f(a) for a in t.axis], t.idx, t.halfwidth, t.null_mask, t.K))
    ctx = B.Context(W.BERRY4, seed=5, K_max=16384)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(25)]
    for e0, e1 in ev:
        e0.record()
        ctx.step(dt, 0.15, 0.01, 0.025)
        e1.record()
    torch.cuda.synchronize()
    assert np.median([e0.elapsed_time(e1) for e0, e1 in ev[5:]]) * 1e3 < 1.2 * us
