"""The randomised two-arm calibration by candidates (csrc/sim_tail.cu) where the cap on
the selection is itself a table value: S(0, 2) = S(1, 4) = S(4, 8) for n = 16, but their
differences x_1 - x_0 are 2, 3 and 4, and trials with S below that value have at least 3.
Success rates are stepped one float at a time, so that the cap passes over the value;
every output agrees bit for bit with the cell histogram and its tie pass, which see
every trial."""
import dataclasses
import math
from statistics import NormalDist

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


@pytest.mark.parametrize("alpha", [0.0590, 0.0597, 0.0604])
def test_cap_on_a_value_that_cells_of_different_difference_share(B, alpha):
    n, K, q0 = 16, 16384, 0.13
    tie = (1 - 4) / n / math.sqrt(5.0 / 32.0 * 27.0 / 32.0 * 2.0 / n)   # S(1, 4)
    ks = math.floor((K + 1) * alpha)
    z = NormalDist().inv_cdf((ks + 3.0 * math.sqrt(ks) + 1.0) / K)
    # the kernel's cap is (q0 - q1) den + z sd + 0.05 with sd near 1: the q1 that brings it to the value
    q1 = q0
    for _ in range(50):
        pb = 0.5 * (q0 + q1)
        den = 1.0 / math.sqrt(pb * (1.0 - pb) * 2.0 / n)
        sd = math.sqrt((q0 * (1.0 - q0) + q1 * (1.0 - q1)) / n) * den
        q1 = q0 - (tie - 0.05 - z * sd) / den
    step = 2.0 ** -26   # floats near 0.13
    logit = lambda q: np.log(q / (1.0 - q))
    ax = [logit(float(np.float32(q)) + step * np.arange(-64, 64)) for q in (q0, q1)]
    i0, i1 = np.meshgrid(np.arange(128), np.arange(128), indexing="ij")
    idx = np.stack([i0.ravel(), i1.ravel()], axis=1).astype(np.int32)
    tiles = W.TileSet(2, ax, idx, np.zeros((idx.shape[0], 2)), np.ones(idx.shape[0], np.uint32),
                      np.full(idx.shape[0], K, np.int32))
    dt = B.DeviceTiles(tiles)
    ctx = B.Context(dataclasses.replace(W.TWO_ARM, looks=(n,)), seed=3, K_max=K)
    a = ctx.calibrate_rand(dt, alpha)
    ctx.set_option(B.OPT_SIM_THREADS, 128)
    b = ctx.calibrate_rand(dt, alpha)
    torch.cuda.synchronize()
    ctx.sync()
    # the order statistic is the value, on which the cap lies for some of the tiles
    assert abs(b["lambda_tile"].median().item() - tie) < 1e-6
    for k in ("lambda_tile", "c_tile"):
        assert torch.equal(a[k], b[k]), (k, int((a[k] != b[k]).sum()))
    assert (a["lam"], a["c"]) == (b["lam"], b["c"])
