"""The count tables (csrc/uniforms.cu): success counts read back through the exported
statistics (one arm: S is strictly falling in the count, so equal S means equal
counts) and through the exact integers of the simulation, for axis values that rise,
fall and repeat, more than one chunk of values, values outside every uniform, K
around the block of 128 sims, and patients at the edges of a Philox block."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _axis(order, n, seed):
    rng = np.random.default_rng(seed)
    v = np.concatenate([rng.uniform(-4.0, 4.0, n - 6), [-800.0, 800.0, -40.0, 40.0, 0.0, 0.0]])
    return {"rising": np.sort(v), "falling": np.sort(v)[::-1].copy(), "mixed": rng.permutation(v)}[order]


@pytest.mark.parametrize("order", ["rising", "falling", "mixed"])
@pytest.mark.parametrize("n,n_axis,K", [(1, 31, 1), (5, 512, 127), (50, 513, 129), (127, 1100, 300), (128, 40, 1041)])
def test_one_arm_counts(B, order, n, n_axis, K):
    design = dataclasses.replace(W.ONE_ARM, looks=(n,), seed=11)
    ax = _axis(order, n_axis, n)
    tiles = W.TileSet(1, [ax], np.arange(n_axis, dtype=np.int32)[:, None], np.full((n_axis, 1), 0.01),
                      np.ones(n_axis, np.uint32), np.full(n_axis, K, np.int32))
    ctx = B.Context(design, K_max=K + 7)
    S, off = ctx.statistics(B.DeviceTiles(tiles))
    torch.cuda.synchronize()
    ctx.sync()
    ref = O.simulate(design, tiles, 0.0, want_S=True)["S"]
    assert np.array_equal(S.cpu().numpy(), np.concatenate(ref).astype(np.float32))


@pytest.mark.parametrize("looks", [(1, 2, 3), (10, 20, 40), (20, 40, 70)])
def test_multi_look_counts(B, looks):
    """Three look segments, interim counts in nibbles and in planes of their own: the
    basket and selection designs' success sums against the oracle's integers."""
    design = W.Design("bayes4", "bayes4", 4, looks, seed=4)
    rng = np.random.default_rng(7)
    n = 60
    ax = [rng.permutation(np.linspace(-2.0, 2.0, 270)) for _ in range(4)]
    tiles = W.TileSet(4, ax, rng.integers(0, 270, (n, 4)).astype(np.int32), np.full((n, 4), 0.01),
                      rng.integers(1, 8, n).astype(np.uint32), rng.integers(1, 400, n).astype(np.int32))
    ctx = B.Context(design, K_max=400)
    R, X, _ = ctx.simulate_tiles(B.DeviceTiles(tiles), 0.3)
    torch.cuda.synchronize()
    ctx.sync()
    ref = O.simulate(design, tiles, 0.3)
    same = R.cpu().numpy() == ref["R"]              # FP32 against FP64 posterior: rare flips
    assert same.mean() > 0.95
    assert np.array_equal(X.cpu().numpy()[same], ref["Xrej"][same])
