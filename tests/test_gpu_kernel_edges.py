"""Kernels of the round loop at the sizes where their tilings, passes and dispatch rules change, against the oracle at the
tolerances of the parity tests."""
import numpy as np
import pytest

from conftest import make_oracle
from helpers import compare_with_oracle, oracle_run_with_paths
from oracle import models
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


@pytest.mark.parametrize("B", [12, 13])
def test_local_steps_few_rows_of_a_large_model(B):
    """One CTA per worker up to 12 rows, clusters above."""
    cfg = _small_cfg(inputs.SOFTMAX, (784, 10), inputs.BF16, 100, B, 100, 5, GAMMA3, lr=0.005)
    X, y, w0 = _problem(cfg)
    compare_with_oracle(cfg, X, y, w0, 4, TOL_BF16, forced=True, loss_tol=5e-2, local_steps=3)


# Least-squares runs from a w0 of the size of the generating weights, so that x.w weighs as much as y in every residual.
# Binary32 sums leave losses and path at 1e-6.  From round 1 on a stored weight (of size 1) may lie on the other side of a bf16
# rounding, 2^-8 away; n of those change a residual of size sqrt(2 d) by about sqrt(n) 2^-8, a loss by 2 sqrt(n) 2^-8 / sqrt(2 d):
# 7e-4 for 64 of 4096.  Their number grows fivefold a round once there is one, hence three rounds (seen: 1, and 2e-5).
LSQ_LOSS_TOL = 1e-3
LSQ_MOVE_TOL = 1e-3


def _without_last_columns(w, Xb, yb):
    """models.lsq_loss_grad, but the dot products miss the last 16 bytes of a row."""
    r = Xb[:, :-8] @ w[:-8] - yb if len(w) > 8 else -yb
    return 0.5 * np.mean(r * r), (Xb.T @ r) / Xb.shape[0]


@pytest.mark.parametrize("d,B,K0", [
    # one or two items per CTA
    (8, 9, 150), (2040, 13, 150),                              # one column slice per thread
    (2048, 4, 150), (2056, 5, 150), (4096, 1, 150), (4096, 3, 150), (4088, 16, 150),      # ... two; rows for one team only
    # the producer holds four items' rows at a time; items per CTA on 148 SMs:
    (4096, 16, 297), (64, 16, 297),                            # 4 or 5
    (4096, 32, 297), (2048, 32, 297),                          # 8 or 9
    (4096, 33, 297), (72, 33, 297),                            # 10 or 11, the last of a worker with one row
    (4096, 61, 297), (64, 61, 297),                            # 16 or 17, the last of a worker with a row for the second team
])
def test_least_squares_pipeline_teams(d, B, K0, monkeypatch):
    lr = 0.3 / ((1 + (d / (K0 * B)) ** 0.5) ** 2 * (1 + 300 / K0))
    cfg = _small_cfg(inputs.LSQ, (d, 1), inputs.BF16, 300, B, K0, 6, GAMMA3, lr=lr)
    X, y, _ = _problem(cfg)
    w0 = np.random.default_rng(17).standard_normal(d).astype(np.float32)
    rows, orows, _, o = compare_with_oracle(cfg, X, y, w0, 3, TOL_BF16, k_mode=gpu.K_FIXED, loss_tol=LSQ_LOSS_TOL,
                                           move_tol=LSQ_MOVE_TOL)
    # what the comparison can see: one missing 16-byte slice of the dot products
    monkeypatch.setattr(models, "lsq_loss_grad", _without_last_columns)
    bad = make_oracle(cfg, X, y, w0, k_mode=gpu.K_FIXED)
    brows, path = oracle_run_with_paths(cfg, bad, 3)
    a, b = (np.array(r[0]["sel_loss"]) for r in (orows, brows))
    assert np.mean(np.abs(a - b) > LSQ_LOSS_TOL * a) > 0.9
    assert np.linalg.norm(bad.w - o.w) > 10 * LSQ_MOVE_TOL * path["w"]
