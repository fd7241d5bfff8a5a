"""Kernels of the round loop at the sizes where their tilings, passes and dispatch rules change, against the oracle at the
tolerances of the parity tests."""
import pytest

from helpers import compare_with_oracle
from paper_2301_08895_b200 import abs as gpu
from paper_2301_08895_b200 import inputs
from test_gpu_parity import GAMMA3, PARETO, TOL_BF16, TOL_FP32, _problem, _small_cfg

pytestmark = pytest.mark.gpu

CONST = inputs.TimeSpec(kind=inputs.T_CONST, shift=1.0)


@pytest.mark.parametrize("W", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257])
@pytest.mark.parametrize("time", [GAMMA3, CONST], ids=["gamma", "ties"])
def test_control_step_worker_counts(W, time):
    """Ranks by counting (8, 4, 2 lanes per key), by merging, 1024 threads; loss sums of one and of several warps; equal ticks."""
    cfg = _small_cfg(inputs.SOFTMAX, (12, 3), inputs.FP32, W, 5, max(1, W // 3), 5, time, lr=0.02)
    X, y, w0 = _problem(cfg)
    compare_with_oracle(cfg, X, y, w0, 25, TOL_FP32, forced=True)


@pytest.mark.parametrize("W,K0,S,B", [
    (90, 2, 70, 3),        # staleness groups beyond 32 and 64
    (24, 24, 3, 85),       # 2040 rows and padding: more row losses than the step fetches ahead of time
    (300, 100, 6, 13),     # ... with 1024 threads
])
def test_control_step_row_layouts(W, K0, S, B):
    cfg = _small_cfg(inputs.SOFTMAX, (12, 3), inputs.FP32, W, B, K0, S, PARETO, lr=0.01)
    X, y, w0 = _problem(cfg)
    compare_with_oracle(cfg, X, y, w0, 60 if W == 90 else 15, TOL_FP32, forced=True, k_mode=gpu.K_FIXED)


@pytest.mark.parametrize("dims,W,B,U", [
    ((40, 6), 6, 150, 2),        # one CTA per worker: soft-max of its rows in three passes
    ((128, 16), 5, 300, 2),      # four: 75 rows each, two passes
    ((784, 10), 17, 20, 2),      # eight, more clusters than have an SM per CTA; the last owner has two rows of three
])
def test_local_steps_rows_per_owner(dims, W, B, U):
    cfg = _small_cfg(inputs.SOFTMAX, dims, inputs.FP32, W, B, 3, 5, GAMMA3, lr=0.02)
    X, y, w0 = _problem(cfg)
    compare_with_oracle(cfg, X, y, w0, 6, TOL_FP32, forced=True, local_steps=U)


@pytest.mark.parametrize("d,B", [(8, 9), (2040, 13), (2048, 4), (2056, 5), (4096, 1), (4096, 3), (4088, 16)])
def test_least_squares_pipeline_teams(d, B):
    """Rows for one team only, one column slice per thread, items more than the first four of a CTA."""
    cfg = _small_cfg(inputs.LSQ, (d, 1), inputs.BF16, 300, B, 150, 6, GAMMA3, lr=0.02 / d)
    X, y, w0 = _problem(cfg)
    compare_with_oracle(cfg, X, y, w0, 6, TOL_BF16, forced=True, loss_tol=5e-2)
