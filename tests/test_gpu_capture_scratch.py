"""Selection keys and CUDA graphs: a step that needs more key scratch than the calls
before it reserved is captured all the same (fewer blocks, or the cell histogram, which
needs none), as nothing may be allocated during a capture; so is the first call of the
plain path; and a captured step keeps its scratch when a later call of the same context
needs more."""
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu
KEYS = ("R", "Xrej", "lambda_tile", "lam", "u0", "bound")


@pytest.fixture(scope="module")
def B():
    from paper_2212_10042_gb300 import binding
    binding.lib()
    return binding


def _capture(ctx, dt, lam, alpha, out):
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        ctx.step(dt, lam, 0.01, alpha, out)
    torch.cuda.current_stream().wait_stream(side)
    return graph


def _replayed(graph, out):
    for k in KEYS:
        out[k].zero_()
    graph.replay()
    torch.cuda.synchronize()
    return {k: out[k].clone() for k in KEYS}


@pytest.mark.parametrize("design,tiles,K_before,alpha_before", [
    (W.TWO_ARM, lambda K: W.two_arm_grid(40, K), 3000, 0.3),          # the cell histogram before: no keys
    (W.TWO_ARM, lambda K: W.two_arm_grid(110, K), 65552, 0.025),      # two tiles a block before, four now
    (W.BAYES4, lambda K: W.four_arm_grid(7, K), (1 << 17) + 16, 0.025),
])
def test_step_that_needs_more_keys_is_captured(B, design, tiles, K_before, alpha_before):
    K = min(K_before, 65536)
    lam = 0.06 if design is W.BAYES4 else -1.96
    ctx = B.Context(design, seed=9, K_max=K_before)
    ctx.step(B.DeviceTiles(tiles(K_before)), lam, 0.01, alpha_before)
    dt = B.DeviceTiles(tiles(K))
    out = ctx.step_buffers(dt)
    got = _replayed(_capture(ctx, dt, lam, 0.025, out), out)
    ref = B.Context(design, seed=9, K_max=K_before).step(dt, lam, 0.01, 0.025)
    torch.cuda.synchronize()
    for k in KEYS:
        assert torch.equal(got[k], ref[k]), k


def test_plain_call_is_captured(B):
    """The sorted uniforms of the plain path are there before its first call."""
    dt = B.DeviceTiles(W.two_arm_grid(12, 700))
    ctx = B.Context(W.TWO_ARM, seed=9, K_max=700)
    out = ctx.step_buffers(dt)
    ref = {k: v.clone() for k, v in ctx.step(dt, -1.96, 0.01, 0.025, out).items() if k in KEYS}
    ctx.set_option(B.OPT_PLAIN, 1)
    got = _replayed(_capture(ctx, dt, -1.96, 0.025, out), out)
    for k in ("R", "Xrej", "lambda_tile", "lam"):
        assert torch.equal(got[k], ref[k]), k


def test_captured_step_outlives_a_call_with_more_keys(B):
    """The randomised calibration takes keys of twice the size."""
    dt = B.DeviceTiles(W.two_arm_grid(64, 9000))
    ctx = B.Context(W.TWO_ARM, seed=9, K_max=9000)
    out = ctx.step_buffers(dt)
    ref = {k: v.clone() for k, v in ctx.step(dt, -1.96, 0.01, 0.025, out).items() if k in KEYS}
    graph = _capture(ctx, dt, -1.96, 0.025, out)
    ctx.calibrate_rand(dt, 0.025)
    filler = [torch.zeros(1 << 24, dtype=torch.uint8, device="cuda") for _ in range(8)]   # takes freed memory, if any
    torch.cuda.synchronize()
    got = _replayed(graph, out)
    assert all(int(f.count_nonzero()) == 0 for f in filler)
    for k in KEYS:
        assert torch.equal(got[k], ref[k]), k
