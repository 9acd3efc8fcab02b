"""The Clopper-Pearson solve by groups of lanes (csrc/bound.cu) against the binomial tail
summed in extended precision, up to K = 2^20 and confidence levels near one half, where
the continued fraction needs several passes.

The tolerance.  The log of the tail is a sum of terms up to |e| <= 4 sd K in FP64, with
log1p and products at one unit in the last place each: an absolute error of at most
8 eps |e|, eps = 1.1e-16.  The tail's derivative in u is at least 0.8 / sd at these levels,
so u is off by at most 1.25 sd (8 eps 4 sd K) = 40 eps sd^2 K = 40 eps u (1 - u), that is
40 eps relative; the Halley step adds less than eps."""
import math

import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu
RTOL = 41 * 2.0 ** -53
LD = np.longdouble


def _deviance(x, m):   # x log(x / m) + m - x, |x - m| << x + m (C. Loader 2000)
    d = x - m
    v = d / (x + m)
    s, t = d * v, LD(2) * x * v
    for j in range(1, 60):
        t = t * v * v
        s = s + t / LD(2 * j + 1)
    return s


def _stirling(n):
    r = LD(1) / n
    return r * (LD(1) / 12 - r * r * (LD(1) / 360 - r * r * (LD(1) / 1260 - r * r * (LD(1) / 1680 - r * r / LD(1188)))))


def _relative_error(R, K, u, delta):
    """(u - exact) / u to first order: one Newton step of log P(Binom(K, u) <= R) - log delta."""
    n, r, u = LD(K), LD(R), LD(u)
    lt = (_stirling(n) - _stirling(r) - _stirling(n - r) - _deviance(r, n * u) - _deviance(n - r, n * (1 - u))
          + LD(0.5) * np.log(n / (2 * LD(math.pi) * r * (n - r))))   # log of the term at R
    j = np.arange(min(R, 12000), dtype=LD)
    tail = LD(1) + np.cumprod((r - j) / (n - r + j + 1) * ((1 - u) / u)).sum()
    f = lt + np.log(tail) - np.log(LD(delta))
    pdf_over_tail = (n - r) / ((1 - u) * tail)
    return float(f / pdf_over_tail / u)


@pytest.mark.parametrize("delta", [0.5, 0.45, 0.3, 0.1, 0.01])
def test_upper_bound_at_rounding(delta):
    from paper_2212_10042_gb300 import binding as B

    # two success rates (n = 1 patient a trial has S < 0 iff it succeeds) and K up to 2^20
    rng = np.random.default_rng(8)
    n = 64
    K = np.concatenate([[1 << 20] * 16, np.exp(rng.uniform(math.log(2000), math.log(1 << 20), n - 16))]).astype(np.int32)
    theta = rng.choice([-1.4, -0.2, 0.0, 0.8], n)[:, None]
    tiles = W.from_centers(theta, 0.001, np.ones(n, np.uint32), K)
    design = W.Design("o", "one_arm_z", 1, (1,))
    ctx = B.Context(design, seed=4, K_max=1 << 20)
    out = ctx.validate(B.DeviceTiles(tiles), 0.0, delta)
    torch.cuda.synchronize()
    ctx.sync()
    R, u = out["R"].cpu().numpy(), out["u0"].cpu().numpy()
    assert (R > 100).all() and (R < tiles.K - 100).all()
    # math.pi in LD's own digits is not needed: an error of 1e-16 in the log of the term moves u
    # by 1e-16 sd, below 1e-18 of u
    err = [_relative_error(int(R[i]), int(tiles.K[i]), u[i], delta) for i in range(n)]
    assert max(map(abs, err)) <= RTOL, max(map(abs, err))
