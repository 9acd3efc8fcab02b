"""Two-arm selections over the whole range of response rates (csrc/sim_tail.cu): rates
near 0 or 1, where a large share of the trials were candidates or the normal quantile
misses, alternatives where nearly every trial rejects, very few patients.  Every output
agrees bit for bit with the cell histogram, and the simulation takes hardly longer than
it (with the least difference over all rows, rejections as candidates and repeats by
fixed steps of the cap it took 2 to 9 times as long)."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (patients, lowest and highest theta_0, theta_1 - theta_0)
RANGES = [(100, 1.0, 4.0, 0.0), (57, 3.0, 5.0, 0.0), (57, -6.0, -5.0, 0.0), (100, -1.0, 1.0, 2.0), (5, -3.0, 3.0, 0.0)]


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _tiles(lo, hi, gap, n_tiles, K, seed):
    rng = np.random.default_rng(seed)
    ax = np.linspace(lo, hi, 64)
    i = rng.integers(0, 64, (n_tiles, 2)).astype(np.int32)
    return W.TileSet(2, [ax, ax + gap], i, np.full((n_tiles, 2), 0.01), np.ones(n_tiles, np.uint32),
                     K[rng.integers(0, len(K), n_tiles)].astype(np.int32))


def _context(B, n, K_max, cells):
    ctx = B.Context(dataclasses.replace(W.TWO_ARM, looks=(n,)), seed=11, K_max=K_max)
    if cells:
        ctx.set_option(B.OPT_SIM_THREADS, 128)
    return ctx


@pytest.mark.parametrize("n_tiles", [1, 300, 6000])
@pytest.mark.parametrize("n,lo,hi,gap", RANGES + [(100, -7.0, 7.0, 0.0), (24, -4.0, 4.0, 0.0), (128, -4.0, 4.0, -0.5)])
def test_outputs_over_all_rates(B, n, lo, hi, gap, n_tiles):
    K = np.array([1, 31, 40, 500, 2048, 2049, 4100, 9000, 20011])
    tiles = _tiles(lo, hi, gap, n_tiles, K, n)
    dt = B.DeviceTiles(tiles)
    out = []
    for cells in (False, True):
        ctx = _context(B, n, 20011, cells)
        got = []
        for _ in range(2):   # the second call finds the queue and the list's count as the first left them
            for lam, alpha in ((-1.96, 0.025), (-1.0, 0.1), (-3.0, 0.001)):
                s = ctx.step(dt, lam, 0.01, alpha)
                got += [s[k].clone() for k in ("R", "Xrej", "score", "lambda_tile", "lam", "u0")]
                r = ctx.calibrate_rand(dt, alpha)
                got += [r["lambda_tile"], r["c_tile"], torch.tensor([r["lam"], float(r["c"])])]
                c = ctx.calibrate(dt, alpha)
                got += [c["lambda_tile"], torch.tensor(c["lam"])]
        torch.cuda.synchronize()
        ctx.sync()
        out.append(got)
    for j, (x, y) in enumerate(zip(*out)):
        assert torch.equal(x, y), j


@pytest.mark.parametrize("n,lo,hi,gap", RANGES)
def test_no_slower_than_the_cell_histogram(B, n, lo, hi, gap):
    tiles = _tiles(lo, hi, gap, 8192, np.array([16384]), 3)
    dt = B.DeviceTiles(tiles)
    for rand in (False, True):
        ms = []
        for cells in (False, True):
            ctx = _context(B, n, 16384, cells)
            call = (lambda: ctx.calibrate_rand(dt, 0.025)) if rand else (lambda: ctx.step(dt, -1.96, 0.01, 0.025))
            for _ in range(3):
                call()
            ctx.profile(True)
            for _ in range(10):
                call()
            p = ctx.profile_read()
            ms.append(sum(p[k][1] for k in ("sim_ztest", "tie_pass") if k in p))
        assert ms[0] < 1.6 * ms[1], (rand, ms)
