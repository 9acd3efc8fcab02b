"""The four-arm simulation at levels that make most trials candidates (csrc/sim_bayes4.cu):
a warp then evaluates all trials of its step from whole count words.  A call takes no
longer than with every trial in a straight line (the outputs at such levels are compared
with the direct form in test_gpu_bayes4_candidates.py)."""
import numpy as np
import pytest
import torch

from paper_2212_10042_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call,level,us", [("validate", 1.0, 570.0), ("calibrate", 0.3, 530.0)])
def test_time_where_most_trials_are_candidates(call, level, us):
    """us: the call with every trial in a straight line, on this grid (8^4, K = 16,384)."""
    from paper_2212_10042_gb300 import binding as B

    dt = B.DeviceTiles(W.four_arm_grid(8, 16384))
    ctx = B.Context(W.BAYES4, seed=5, K_max=16384)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(25)]
    for e0, e1 in ev:
        e0.record()
        ctx.validate(dt, level, 0.01) if call == "validate" else ctx.calibrate(dt, level)
        e1.record()
    torch.cuda.synchronize()
    assert np.median([e0.elapsed_time(e1) for e0, e1 in ev[5:]]) * 1e3 < 1.05 * us
