"""The z-test simulation by byte-parallel counts and by candidates (csrc/sim_tail.cu)
against the cell-histogram kernel and its tie pass (a fixed configuration selects
them), which see every trial:
all outputs are whole numbers or table values and agree bit for bit, for one and two
arms, patients from 2 to 128, K at the edges of words and steps, the three groupings,
tiles whose order statistic lies past the candidates, and thresholds on and between
table values."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EDGES = np.array([1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 1023, 1024, 1025, 1040, 2047, 2049, 5003, 8193])


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _tiles(d, n, K, seed):
    rng = np.random.default_rng(seed)
    ax = np.linspace(-3.0, 3.0, 41)
    c = ax[rng.integers(0, ax.size, (n, d))]
    c[: n // 8] = 2.0 if d == 1 else np.array([-2.0, 2.0])   # far outside the null set: S small throughout
    return W.from_centers(c, 0.02, np.ones(n, np.uint32), K[rng.integers(0, len(K), n)].astype(np.int32))


def _outputs(ctx, dt, lams, alphas):
    out = []
    for lam in lams:
        out += [x.clone() for x in ctx.simulate_tiles(dt, lam)]
        for c in (0, 1 << 30, 0xFFFFFFFF):
            v = ctx.validate_rand(dt, lam, c, 0.01)
            out += [v[k].clone() for k in ("R", "Xrej", "score")]
    for alpha in alphas:
        s = ctx.step(dt, lams[0], 0.01, alpha)
        out += [s[k].clone() for k in ("R", "Xrej", "score", "lambda_tile", "lam")]
        cal = ctx.calibrate(dt, alpha)
        out += [cal["lambda_tile"].clone(), torch.tensor(cal["lam"])]
        r = ctx.calibrate_rand(dt, alpha)
        out += [r["lambda_tile"].clone(), r["c_tile"].clone(), torch.tensor([r["lam"], float(r["c"])])]
    torch.cuda.synchronize()
    ctx.sync()
    return out


def _compare(B, design, tiles, lams, alphas):
    ctx = B.Context(design, seed=21, K_max=int(tiles.K.max()))
    dt = B.DeviceTiles(tiles)
    a = _outputs(ctx, dt, lams, alphas)
    ctx.set_option(B.OPT_SIM_THREADS, 128)
    b = _outputs(ctx, dt, lams, alphas)
    for j, (x, y) in enumerate(zip(a, b)):
        assert torch.equal(x, y), j


@pytest.mark.parametrize("n_tiles", [60, 1300, 4900])
@pytest.mark.parametrize("stat,n", [("one", 50), ("one", 128), ("two", 2), ("two", 57), ("two", 100), ("two", 126), ("two", 128)])
def test_candidates_match_the_cell_histogram(B, stat, n, n_tiles):
    design = dataclasses.replace(W.ONE_ARM if stat == "one" else W.TWO_ARM, looks=(n,))
    tiles = _tiles(design.d, n_tiles, EDGES, n)
    S = torch.unique(B.Context(design, K_max=2048).statistics(B.DeviceTiles(_tiles(design.d, 64, EDGES[:16], 1)))[0])
    on = S[S <= -1.0]
    lams = (-1.96, -1.0, -40.0, 0.0, float("inf")) + ((float(on[len(on) // 2]),) if len(on) else ())
    _compare(B, design, tiles, lams, (0.025, 0.001))


@pytest.mark.parametrize("K", [70000, 1 << 18, 300000, 1 << 20])
def test_candidates_at_large_K(B, K):
    tiles = _tiles(2, 9, np.array([K, K - 1, 65537]), 5)
    _compare(B, W.TWO_ARM, tiles, (-1.96,), (0.025,))
