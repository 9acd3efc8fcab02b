"""Measured cases of the CSE hot path.

A case is one call (or one short sequence of calls) that a user of this package
makes through `paper_2212_10042_gb300.binding` / `.adaptive`, at sizes of the
package's own workloads, tests and benchmark:

  step            reseed + cse_step + score backward: one new batch of
                  simulations, validated and calibrated (the benchmark's step)
  validate, band  cse_validate / cse_validate_band at fixed simulations
  calibrate_rand  cse_calibrate_rand (the randomised z-tests)
  adaptive        GpuCalibrator on a host tile set: one round of the adaptive
                  loop, which uploads a new platten and reads its result back
  gradient        TypeIError forward and backward at free points

`design` with `looks` is the trial, `tiles` the tile set (a null-space grid, a
mixed-level batch, a refined platten, or free points), `K_min` .. `K_max` the
simulations of a tile (log-uniform and ragged where they differ).
"""
import math

import numpy as np
import torch

from paper_2212_10042_gb300 import workloads as W

LAMBDA = {"one_arm_z": -1.96, "two_arm_pooled_z": -1.96, "bayes4": 0.06, "berry4": 0.15}
ARMS = {"one_arm_z": 1, "two_arm_pooled_z": 2, "bayes4": 4, "berry4": 4}
DELTA, ALPHA = 0.01, 0.025
MAX_SIMS = {"one_arm_z": 2 ** 28, "two_arm_pooled_z": 2 ** 33, "bayes4": 2 ** 34, "berry4": 2 ** 34}


def _case(call, design, looks, tiles, size, K_min, K_max, name=None):
    c = dict(call=call, design=design, looks=",".join(map(str, looks)), tiles=tiles, size=size, K_min=K_min,
             K_max=K_max)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one tile row of a single-arm z-test (benchmark configuration c1): the
        # smallest call, where launches and the serial chain of small kernels count
        _case("step", "one_arm_z", (50,), "grid", 64, 8192, 8192, "one_arm_step"),
        # many small tiles with ragged K, R from 0 up: the validation of a fine
        # one-arm grid, hundreds of distinct (K, R) for the Clopper-Pearson solve
        _case("validate", "one_arm_z", (50,), "grid", 1500, 300, 65536, "one_arm_validate_ragged"),
        # the two-arm z-test on the 256 x 256 grid (c2): the ordinary platten
        _case("step", "two_arm_pooled_z", (100,), "grid", 256, 16384, 16384, "two_arm_step"),
        # the throughput batch of mixed-level tiles with K = 2^12 .. 2^16 (c3)
        _case("step", "two_arm_pooled_z", (100,), "batch", 1 << 18, 1 << 12, 1 << 16, "two_arm_batch_step"),
        # a two-sided validation band on an odd grid, odd patients and odd K
        _case("band", "two_arm_pooled_z", (57,), "grid", 61, 5003, 5003, "two_arm_band_odd"),
        # the randomised two-arm test (pairs of statistic and tie-break word)
        _case("calibrate_rand", "two_arm_pooled_z", (100,), "grid", 128, 16384, 16384, "two_arm_randomised"),
        # the differentiable Type I Error at free points (every coordinate its
        # own), forward and backward, as an optimiser over theta calls it
        _case("gradient", "two_arm_pooled_z", (100,), "points", 2048, 8192, 8192, "two_arm_gradient"),
        # the four-arm Bayesian selection design on the 16^4 grid (c4)
        _case("step", "bayes4", (10, 20, 40), "grid", 16, 1 << 14, 1 << 14, "four_arm_step"),
        # the same design on an adaptively refined platten at K = 2^16: a quarter
        # of the benchmark's default workload (c5), the largest work here
        _case("step", "bayes4", (10, 20, 40), "refined", 1 << 18, 1 << 16, 1 << 16, "four_arm_refined_step"),
        # one round of the adaptive loop: a few thousand tiles, ragged K, host
        # buffers in and out
        _case("adaptive", "bayes4", (10, 20, 40), "refined", 60000, 2048, 65536, "four_arm_adaptive"),
        # the basket trial on its 16^4 grid
        _case("step", "berry4", (35,), "grid", 16, 1 << 14, 1 << 14, "basket_step"),
        # validation only (no order statistic) of the basket trial, coarse grid
        # and ragged K
        _case("validate", "berry4", (35,), "grid", 9, 1000, 30000, "basket_validate_ragged"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any design and call, sizes spread over
    their logarithm, odd sizes included, at most the largest listed work."""
    design = rng.choice(["one_arm_z", "two_arm_pooled_z", "two_arm_pooled_z", "bayes4", "bayes4", "berry4"])
    K_max = _log_int(rng, 500, 65536)
    K_min = K_max if rng.random() < 0.5 else max(64, K_max // rng.choice([2, 5, 16]))
    if design == "one_arm_z":
        looks = (_log_int(rng, 20, 128),)
        tiles, size = "grid", _log_int(rng, 16, 4096)
        call = rng.choice(["step", "validate", "band", "calibrate_rand", "gradient"])
    elif design == "two_arm_pooled_z":
        looks = (_log_int(rng, 20, 128),)
        tiles = rng.choice(["grid", "batch"])
        size = _log_int(rng, 8, 256) if tiles == "grid" else _log_int(rng, 64, 1 << 18)
        call = rng.choice(["step", "validate", "band", "calibrate_rand", "adaptive", "gradient"])
    elif design == "bayes4":
        # the last of these has final-look codes beyond seven bits
        looks = rng.choice([(10, 20, 40), (10, 20, 40), (8, 17, 31), (20, 40, 70)])
        tiles = rng.choice(["grid", "refined"])
        size = _log_int(rng, 4, 15) if tiles == "grid" else _log_int(rng, 52000, 1 << 17)
        call = rng.choice(["step", "validate", "band", "adaptive"])
    else:
        looks = (_log_int(rng, 12, 45),)
        tiles, size = "grid", _log_int(rng, 4, 16)
        call = rng.choice(["step", "validate", "band"])
    if call == "gradient":
        tiles, size = "points", _log_int(rng, 64, 2048)
        K_max = min(K_max, 16384)
        K_min = K_max
    c = _case(call, design, looks, tiles, size, K_min, K_max)
    while _tile_count(c) * K_max > MAX_SIMS[design]:
        K_max = max(500, K_max // 2)
        c["K_max"], c["K_min"] = K_max, min(c["K_min"], K_max)
    return c


def _tile_count(case):
    """Tiles of the case, from its sizes (the two-dimensional and four-dimensional
    grids keep the boxes that meet a null hypothesis)."""
    n = case["size"]
    if case["tiles"] != "grid":
        return n
    if case["design"] == "two_arm_pooled_z":
        return n * (n + 1) // 2
    if case["design"] == "one_arm_z":
        return n
    return int(n ** 4 * (0.78 if case["design"] == "bayes4" else 0.92))


def _design(case):
    looks = tuple(int(x) for x in case["looks"].split(","))
    null = W.BERRY4.arm_null if case["design"] == "berry4" else (0.0,) * 4
    return W.Design(case["design"], case["design"], ARMS[case["design"]], looks, arm_null=null)


def _tiles(case, seed):
    """The case's tile set; the domain's edges (where the tile count does not depend on
    them), the random centres and the ragged K vary with the seed."""
    rng = np.random.Generator(np.random.PCG64([seed, 17]))
    K, size = case["K_max"], case["size"]
    shift = float(rng.uniform(-0.05, 0.05))
    if case["design"] == "one_arm_z":
        t = W.one_arm_tiles(size, K, lo=-2.0 + shift)
    elif case["design"] == "two_arm_pooled_z":
        if case["tiles"] == "grid":
            t = W.two_arm_grid(size, K, lo=-2.0 + shift, hi=2.0 + shift)
        else:
            t = W.two_arm_adaptive(size, seed=seed, lo=-2.0, hi=2.0)
    elif case["design"] == "bayes4":
        if case["tiles"] == "grid":
            t = W.four_arm_grid(size, K, lo=W.LOGIT_LO + shift, hi=W.LOGIT_HI + shift)
        else:
            # refinement splits whole tiles: cut to the same number for every seed
            t = W.four_arm_refined(size, K, seed=seed).subset(np.arange(size))
    else:
        t = W.berry_grid(size, K)
    if case["K_min"] == K:
        return t.with_K(K)
    n = t.n_tiles
    if case["tiles"] == "batch":   # powers of two, as the adaptive loop's doubling leaves them
        steps = int(math.log2(K / case["K_min"]))
        return t.with_K(K >> rng.integers(0, steps + 1, n))
    return t.with_K(np.exp(rng.uniform(math.log(case["K_min"]), math.log(K + 0.5), n)).astype(np.int32))


def _points(case, seed):
    rng = np.random.Generator(np.random.PCG64([seed, 23]))
    d = ARMS[case["design"]]
    return rng.uniform(-1.5, 0.5, (case["size"], d)), rng.normal(size=case["size"])


def prepare(case, seed):
    from paper_2212_10042_gb300 import adaptive, binding as B

    design, call = _design(case), case["call"]
    st = dict(call=call, lam=LAMBDA[case["design"]], seed=1000 + seed, K=case["K_max"])
    if call == "adaptive":
        st["tiles"] = _tiles(case, seed)
        st["calibrator"] = adaptive.GpuCalibrator(design, ALPHA, case["K_max"], seed=st["seed"])
        return st
    st["ctx"] = B.Context(design, seed=st["seed"], K_max=case["K_max"])
    if call == "gradient":
        theta, g = _points(case, seed)
        st["theta"] = torch.from_numpy(theta).cuda().requires_grad_(True)
        st["g"] = torch.from_numpy(g).cuda()
        return st
    tiles = _tiles(case, seed)
    st["tiles"] = B.DeviceTiles(tiles)
    if call == "step":
        rng = np.random.Generator(np.random.PCG64([seed, 29]))
        st["out"] = st["ctx"].step_buffers(st["tiles"])
        st["g"] = torch.from_numpy(rng.normal(size=tiles.n_tiles)).cuda()
    return st


def run(st):
    from paper_2212_10042_gb300 import binding as B

    call, lam = st["call"], st["lam"]
    if call == "adaptive":
        return st["calibrator"](st["tiles"])
    ctx = st["ctx"]
    if call == "step":
        ctx.reseed(st["seed"])
        out = ctx.step(st["tiles"], lam, DELTA, ALPHA, st["out"])
        return dict(out, grad=B.score_backward(st["g"], out["score"], st["tiles"].K))
    if call == "validate":
        return ctx.validate(st["tiles"], lam, DELTA)
    if call == "band":
        return ctx.validate_band(st["tiles"], lam, DELTA)
    if call == "calibrate_rand":
        return ctx.calibrate_rand(st["tiles"], ALPHA)
    f = B.TypeIError.apply(st["theta"], ctx, 1, st["K"], lam)
    (grad,) = torch.autograd.grad(f, st["theta"], st["g"])
    return dict(f=f.detach(), grad=grad)


def work(case):
    """Bytes: the tile set read once, every output written once.  Operations: one
    per arm for each (tile, simulation) (the trial's outcome read), Philox's 40
    multiplies and xors a counter block where the call draws new uniforms, and
    about 10 evaluations of 30 operations per arm and sign for each q-search."""
    d, call, n = ARMS[case["design"]], case["call"], _tile_count(case)
    n_max = int(case["looks"].split(",")[-1])
    lo, hi = case["K_min"], case["K_max"]
    mean_K = hi if lo == hi else (hi - lo) / math.log(hi / lo)
    if case["tiles"] == "batch" and lo != hi:
        steps = int(math.log2(hi / lo))
        mean_K = sum(hi >> i for i in range(steps + 1)) / (steps + 1)
    if call == "gradient":
        return dict(bytes=float(n * (8 * d + 8 + 8 + 8 + 8 * d)), flops=float(n * mean_K * d))
    tile_in = 4 * d + 8 * d + 4 + 4
    per_tile = {"step": 8 + 16 * d + 8 * 5 + 8 + 8 * d, "validate": 8 + 16 * d + 24, "band": 8 + 16 * d + 32,
                "calibrate_rand": 20, "adaptive": 16}[call]
    searches = {"step": 2, "validate": 1, "band": 2, "calibrate_rand": 1, "adaptive": 1}[call]
    flops = n * mean_K * d + searches * n * 10 * 2 * d * 30
    if call == "step":
        flops += hi * d * ((n_max + 3) // 4) * 40
    return dict(bytes=float(n * (tile_in + per_tile)), flops=float(flops))


# ---------------------------------------------------------------------------
# The same quantities in plain 64-bit torch, from the method's formulas.
# ---------------------------------------------------------------------------
EXACT_SIMS = 1.2e9   # (tile, simulation) pairs up to which exact() evaluates a case
M32 = 0xFFFFFFFF


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors of 32-bit words."""
    def mul(m, x):
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        return (hi + (lo >> 16)) >> 16, (((hi & 0xFFFF) << 16) + lo) & M32

    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _counts(seed, looks, arm, theta, K):
    """[look][value][K] cumulative success counts of the arm at each value of theta."""
    dev = theta.device
    p = 1.0 / (1.0 + torch.exp(-theta))
    thr = torch.clamp(torch.floor(p * 4294967296.0), 0.0, 4294967295.0).to(torch.int64)
    out = [torch.empty((theta.numel(), K), dtype=torch.uint8, device=dev) for _ in looks]
    n, step = looks[-1], max(1, (1 << 26) // max(theta.numel(), looks[-1]))
    for k0 in range(0, K, step):
        k = torch.arange(k0, min(K, k0 + step), dtype=torch.int64, device=dev)[:, None]
        j = torch.arange((n + 3) // 4, dtype=torch.int64, device=dev)[None, :]
        z = torch.zeros_like(k + j)
        words = torch.stack(_philox(k + z, z + arm, z + j, z, seed), dim=-1).reshape(k.numel(), -1)[:, :n]
        total, prev = 0, 0
        for look, end in enumerate(looks):
            seg = words[:, prev:end].sort(dim=1).values.contiguous()
            total = total + torch.searchsorted(seg, thr.expand(k.numel(), -1).contiguous())
            out[look][:, k0:k0 + k.numel()] = total.to(torch.uint8).T
            prev = end
    return out


def _nodes():
    L = [math.log(1e-6) + (math.log(1e3) - math.log(1e-6)) * j / 15.0 for j in range(16)]
    s2 = [math.exp(x) for x in L]
    lp = [(math.log(0.5) if j in (0, 15) else 0.0) - 1.0005 * L[j] - 0.000005 / s2[j] + L[j] for j in range(16)]
    return s2, lp


def _posterior(x, n, offset, against_control):
    """P(theta_i > theta_0), i = 1..3 (against_control), or 1 - P(theta_i > 0), i =
    0..3, of the hierarchical model, for success counts x of n, [N, 4] tensors."""
    res = []
    for x, n in zip(x.split(1 << 20), n.split(1 << 20)):
        xs, fs = x + 0.5, n - x + 0.5
        th, v0 = torch.log(xs / fs) - offset, 1.0 / xs + 1.0 / fs
        lw, val = [], []
        for s2, lp in zip(*_nodes()):
            den = v0 + s2
            w, r = 1.0 / den, th + 1.34
            Wt = w.sum(1)
            Sr = (w * r).sum(1)
            prec = 0.01 + Wt
            quad = (w * r * r).sum(1) - Sr * Sr / prec
            lw.append(lp - 0.5 * (torch.log(den).sum(1) + torch.log1p(100.0 * Wt)) - 0.5 * quad)
            mu = ((-1.34 * 0.01 + (w * th).sum(1)) / prec)[:, None]
            c, v = v0 * w, v0 * s2 * w
            e = (1.0 - c) * th + c * mu
            if against_control:
                dc = c[:, 1:] - c[:, :1]
                z = (e[:, 1:] - e[:, :1]) / torch.sqrt(v[:, 1:] + v[:, :1] + dc * dc / prec[:, None])
            else:
                z = -e / torch.sqrt(v + c * c / prec[:, None])
            val.append(torch.special.ndtr(z))
        weight = torch.softmax(torch.stack(lw), dim=0)
        res.append((weight[:, :, None] * torch.stack(val)).sum(0))
    return torch.cat(res)


def _grid(dims, dev):
    return torch.stack(torch.meshgrid(*[torch.arange(m, device=dev) for m in dims], indexing="ij"), -1).reshape(
        -1, len(dims))


def _bayes4_stat(looks, drop, dev):
    """S of four-arm trials: a function of counts [look][arm] (equal-shaped int64) and a null mask."""
    n1, n2, n3 = looks
    S2, S3 = n1 + n2 + 2, n1 + n2 + n3 + 3
    f64 = torch.float64
    zero = torch.zeros(4, dtype=f64, device=dev)

    def decode(code):   # treatment code -> (successes, patients) when its data froze
        x = torch.where(code <= n1, code, torch.where(code < S2, code - n1 - 1, code - S2))
        n = torch.where(code <= n1, n1, torch.where(code < S2, n2, n3))
        return x.to(f64), n.to(f64)

    def drops(control, n_control, codes):
        xt, nt = decode(codes)
        x = torch.cat([control[:, None].to(f64), xt], 1)
        n = torch.cat([torch.full_like(x[:, :1], n_control), nt], 1)
        bad = _posterior(x, n, zero, True) < drop
        return (bad * torch.tensor([1, 2, 4], device=dev)).sum(1)

    g = _grid((n1 + 1,) * 4, dev)
    D1 = drops(g[:, 0], n1, g[:, 1:])
    D2 = torch.cat([drops(q[:, 0], n2, q[:, 1:]) for q in _grid((n2 + 1, S2, S2, S2), dev).split(1 << 21)])
    c = torch.arange(S3, device=dev)
    tri = _grid((S3, S3, S3), dev)
    tri = tri[(tri[:, 0] >= tri[:, 1]) & (tri[:, 1] >= tri[:, 2])]   # z >= b >= a, in order of triple index
    T3, T2, NT = c * (c + 1) * (c + 2) // 6, c * (c + 1) // 2, tri.shape[0]
    F = torch.empty(((n3 + 1) * NT, 3), dtype=f64, device=dev)
    xt, nt = decode(tri)
    for x0 in range(n3 + 1):
        x = torch.cat([torch.full_like(xt[:, :1], x0), xt], 1)
        F[x0 * NT:(x0 + 1) * NT] = 1.0 - _posterior(x, torch.cat([torch.full_like(nt[:, :1], n3), nt], 1), zero, True)

    def stat(x, mask):
        d1 = D1[((x[0][0] * (n1 + 1) + x[0][1]) * (n1 + 1) + x[0][2]) * (n1 + 1) + x[0][3]]
        t2 = [torch.where((d1 >> i) & 1 == 1, x[0][i + 1], n1 + 1 + x[1][i + 1]) for i in range(3)]
        d2 = d1 | D2[((x[1][0] * S2 + t2[0]) * S2 + t2[1]) * S2 + t2[2]]
        t3 = torch.stack([torch.where((d2 >> i) & 1 == 1, t2[i], S2 + x[2][i + 1]) for i in range(3)], -1)
        t3, who = t3.sort(dim=-1, descending=True)   # z, b, a
        q = F[x[2][0] * NT + T3[t3[..., 0]] + T2[t3[..., 1]] + t3[..., 2]]
        use = (mask[..., None] & ~d2[..., None]) >> who & 1
        return torch.where(use == 1, q, math.inf).amin(-1)

    return stat


def _statistic(case, design, dev):
    """S of trials from counts [look][arm] and the tile's mask, in FP64."""
    f64, n = torch.float64, design.n_max
    if design.stat == "one_arm_z":
        return lambda x, mask: -(x[0][0].to(f64) - n * design.p0) / math.sqrt(n * design.p0 * (1 - design.p0))
    if design.stat == "two_arm_pooled_z":
        g = _grid((n + 1, n + 1), dev).to(f64)
        pb = (g[:, 0] + g[:, 1]) / (2 * n)
        var = pb * (1 - pb) * (2.0 / n)
        tab = torch.where(var > 0, (g[:, 0] - g[:, 1]) / n / torch.sqrt(torch.where(var > 0, var, 1.0)), 0.0)
        return lambda x, mask: tab[x[0][0] * (n + 1) + x[0][1]]
    if design.stat == "bayes4":
        return _bayes4_stat(design.looks, design.drop, dev)
    m = n + 1
    x = _grid((m,) * 4, dev).to(f64)
    tab = _posterior(x, torch.full_like(x, n), torch.tensor(design.arm_null, dtype=f64, device=dev), False)

    def stat(x, mask):
        q = tab[((x[0][0] * m + x[0][1]) * m + x[0][2]) * m + x[0][3]]
        bit = mask[..., None] >> torch.arange(4, device=dev) & 1
        return torch.where(bit == 1, q, math.inf).amin(-1)

    return stat


def _simulate(case, seed, axis, idx, mask, K, ksel=None):
    """R, Xrej, score per tile and, with ksel, the k-th smallest statistic."""
    dev, design = axis[0].device, _design(case)
    lam, d, K_max = LAMBDA[design.stat], design.d, int(K.max())
    cnt = [_counts(1000 + seed, design.looks, a, axis[a], K_max) for a in range(d)]   # [arm][look][value][K]
    stat, n = _statistic(case, design, dev), K.numel()
    R = torch.zeros(n, dtype=torch.int64, device=dev)
    X = torch.zeros((n, d), dtype=torch.int64, device=dev)
    L = torch.full((n,), -math.inf, dtype=torch.float64, device=dev)
    step = max(1, (1 << 24) // K_max)
    for i0 in range(0, n, step):
        sl = slice(i0, min(n, i0 + step))
        Km = int(K[sl].max())
        x = [[cnt[a][look][idx[sl, a]][:, :Km].to(torch.int64) for a in range(d)] for look in range(len(design.looks))]
        live = torch.arange(Km, device=dev)[None, :] < K[sl][:, None]
        S = torch.where(live, stat(x, mask[sl][:, None].expand(-1, Km)), math.inf)
        rej = S < lam
        R[sl] = rej.sum(1)
        for a in range(d):
            X[sl, a] = (rej * x[-1][a]).sum(1)
        if ksel is not None:
            ks = ksel[sl]
            kth = S.sort(dim=1).values.gather(1, torch.clamp(ks - 1, min=0)[:, None])[:, 0]
            L[sl] = torch.where(ks > 0, kth, -math.inf)
    theta = torch.stack([axis[a][idx[:, a]] for a in range(d)], 1)
    score = X - design.n_max * torch.sigmoid(theta) * R[:, None]
    return R, X, score, L


def _tilt(G, q):
    """Phi(q) = sum over arms of the larger of the two per-arm terms, and its q-derivative."""
    P, dP = 0.0, 0.0
    for th, sp0, h, d1, n in G:
        qv = q[:, None] * h
        y = th + qv
        e = torch.exp(-y.abs())
        r, l1 = e / (1.0 + e), torch.log1p(e)
        phi = n * ((y.clamp(min=0) + l1 - sp0) / q[:, None] - d1)
        hq = torch.where(y >= 0, (sp0 - th) - qv * r - l1, qv * r - l1 + sp0)
        dphi = n * hq / (q * q)[:, None]
        best, j = phi.max(dim=1)
        P, dP = P + best, dP + dphi.gather(1, j[:, None])[:, 0]
    return P, dP


def _arms(axis, idx, hw, n):
    def sp(x):
        return x.clamp(min=0) + torch.log1p(torch.exp(-x.abs()))

    G = []
    for a in range(len(axis)):
        th = axis[a][idx[:, a]][:, None]
        h = torch.stack([hw[:, a], -hw[:, a]], 1)
        G.append((th, sp(th), h, sp(th + h) - sp(th), n))
    return G


def _search(G, lc, inverted):
    """Optimum over s = log q in [0, 40] by bisection on the derivative's sign."""
    lo, hi = torch.zeros_like(lc), torch.full_like(lc, 40.0)
    for _ in range(64):
        s = 0.5 * (lo + hi)
        q = torch.exp(s)
        P, dP = _tilt(G, q)
        below = ((lc - P) + q * (q - 1.0) * dP if inverted else lc / (q * q) + dP) < 0
        lo, hi = torch.where(below, s, lo), torch.where(below, hi, s)
    s = 0.5 * (lo + hi)
    q = torch.exp(s)
    P, _ = _tilt(G, q)
    end = s > 40.0 - 1e-6
    Pinf = sum(torch.maximum(n * (h[:, 0] - d1[:, 0]), -n * d1[:, 1]) for _, _, h, d1, n in G)
    if inverted:
        return torch.where(end, torch.maximum(lc - Pinf, q / (q - 1.0) * (lc - P)), q / (q - 1.0) * (lc - P))
    val = (1.0 - 1.0 / q) * lc + P
    at_inf = end & (lc + Pinf <= val)
    val = torch.where(at_inf, lc + Pinf, val)
    one = (val >= 0) | (s < 1e-12) | (lc >= 0)
    return torch.where(one, 0.0, val), torch.where(one, 1.0, torch.where(at_inf, math.inf, q))


def _stirling_error(n):
    """log n! - [(n + 1/2) log n - n + log(2 pi) / 2] (C. Loader 2000)."""
    r = 1.0 / n.clamp(min=16.0)
    series = r * (1 / 12 - r * r * (1 / 360 - r * r * (1 / 1260 - r * r * (1 / 1680 - r * r / 1188))))
    small = torch.tensor([0.0] + [math.lgamma(k + 1.0) - (k + 0.5) * math.log(k) + k - 0.5 * math.log(2 * math.pi)
                                  for k in range(1, 17)], dtype=torch.float64, device=n.device)
    return torch.where(n < 16, small[n.clamp(max=16).to(torch.int64)], series)


def _deviance(x, m):
    """x log(x / m) + m - x without cancellation near x = m (C. Loader 2000)."""
    d, v = x - m, (x - m) / (x + m)
    s, t = d * v, 2.0 * x * v
    for j in range(1, 40):
        t = t * v * v
        s = s + t / (2 * j + 1)
    return torch.where(v.abs() < 0.1, s, x * torch.log(x / m) + m - x)


def _binom_upper(R, N, ld):
    """u with log P(Binom(N, u) <= R) = ld, for 0 < R < N (doubles) and ld < log(1/2),
    so that u > R / N: safeguarded Newton on the log of the sum of binomial terms
    taken downwards from R (they fall from there on)."""
    lo, hi = R / N, torch.ones_like(R)
    mean = (R + 1.0) / (N + 1.0)
    u = torch.minimum(mean + 2.5 * torch.sqrt(mean * (1 - mean) / (N + 2.0)), 0.5 * (1 + mean))
    j = torch.arange(4096, dtype=torch.float64, device=R.device)
    for _ in range(60):
        ratio = (R[:, None] - j).clamp(min=0) / (N - R)[:, None].add(j + 1) * ((1 - u) / u)[:, None]
        s = 1.0 + torch.cumprod(ratio, 1).sum(1)
        lt = (_stirling_error(N) - _stirling_error(R) - _stirling_error(N - R) - _deviance(R, N * u)
              - _deviance(N - R, N * (1 - u)) + 0.5 * torch.log(N / (2 * math.pi * R * (N - R))))
        f = lt + torch.log(s) - ld
        lo, hi = torch.where(f > 0, u, lo), torch.where(f > 0, hi, u)
        un = u + f * s * (1 - u) / (N - R)
        u = torch.where((un > lo) & (un < hi), un, 0.5 * (lo + hi))
    return u


def _cp_upper(R, K, delta):
    """Upper Clopper-Pearson bound per tile, one solve per distinct (K, R)."""
    keys, inv = torch.unique(torch.stack([K.to(torch.int64), R], 1), dim=0, return_inverse=True)
    N, r = keys[:, 0].double(), keys[:, 1].double()
    u = torch.ones_like(N)
    u = torch.where(r <= 0, -torch.expm1(math.log(delta) / N), u)
    mid = torch.nonzero((r > 0) & (r < N))[:, 0]
    for part in mid.split(1024):
        u[part] = _binom_upper(r[part], N[part], math.log(delta))
    return u[inv]


def exact(case, seed):
    dev, call, design = _device(), case["call"], _design(case)
    f64 = torch.float64
    if call == "gradient":
        theta, g = _points(case, seed)
        n, d, K = case["size"], design.d, case["K_max"]
        axis = [torch.from_numpy(np.ascontiguousarray(theta[:, a])).to(dev) for a in range(d)]
        idx = torch.arange(n, device=dev)[:, None].expand(n, d)
        one = torch.ones(n, dtype=torch.int64, device=dev)
        R, _, score, _ = _simulate(case, seed, axis, idx, one, one * K)
        return dict(f=R / K, grad=torch.from_numpy(g).to(dev)[:, None] * score / K)
    t = _tiles(case, seed)
    if float(t.K.astype(np.float64).sum()) > EXACT_SIMS:
        return None
    axis = [torch.from_numpy(a).to(dev) for a in t.axis]
    idx = torch.from_numpy(t.idx.astype(np.int64)).to(dev)
    hw, K = torch.from_numpy(t.halfwidth).to(dev), torch.from_numpy(t.K.astype(np.int64)).to(dev)
    mask = torch.from_numpy(t.null_mask.astype(np.int64)).to(dev)
    G = _arms(axis, idx, hw, float(design.n_max))
    ap = ksel = None
    if call in ("step", "calibrate_rand", "adaptive"):
        ap = torch.exp(_search(G, torch.full((t.n_tiles,), math.log(ALPHA), dtype=f64, device=dev), True))
        ksel = torch.clamp(torch.floor((K + 1.0) * ap), max=K.double()).to(torch.int64)
    R, X, score, lt = _simulate(case, seed, axis, idx, mask, K, ksel)
    lam = lt.amin() if ksel is not None else None
    if call == "adaptive":
        return ap.cpu().numpy(), lt.cpu().numpy(), float(lam)
    if call == "calibrate_rand":   # the tie-break words are whole numbers, decided by ties of the FP32 statistic
        return dict(alpha_prime=ap, lambda_tile=lt, c_tile=None, lam=float(lam), c=None)
    if call == "band":
        u0 = _cp_upper(R, K, 0.5 * DELTA)
        # lower bound: 1 - l is the upper bound of the failures at the same level
        one_l = _cp_upper(K - R, K, 0.5 * DELTA)
        l0 = torch.where(R == 0, 0.0, 1.0 - one_l)
        lb, _ = _search(G, torch.where(R == 0, 0.0, torch.log(one_l)), False)
        ub, _ = _search(G, torch.log(u0), False)
        return dict(R=R, Xrej=X, score=score, l0=l0, lower=-torch.expm1(lb), u0=u0, upper=torch.exp(ub))
    u0 = _cp_upper(R, K, DELTA)
    lb, q = _search(G, torch.log(u0), False)
    out = dict(R=R, Xrej=X, score=score, u0=u0, bound=torch.exp(lb), qstar=q)
    if call == "step":
        rng = np.random.Generator(np.random.PCG64([seed, 29]))
        g = torch.from_numpy(rng.normal(size=t.n_tiles)).to(dev)
        out.update(alpha_prime=ap, lambda_tile=lt, lam=lam.reshape(1), grad=g[:, None] * score / K[:, None])
    return out
