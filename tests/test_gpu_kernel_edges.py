"""Kernels of the round loop at the sizes where their tilings, passes and dispatch rules change, against the oracle at the
tolerances of the parity tests."""
import pytest

from helpers import compare_with_oracle
from paper_2301_08895_b200 import inputs
from test_gpu_parity import GAMMA3, TOL_FP32, _problem, _small_cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,W,B,U", [
    ((40, 6), 6, 150, 2),        # one CTA per worker: soft-max of its rows in three passes
    ((128, 16), 5, 300, 2),      # four: 75 rows each, two passes
    ((784, 10), 17, 20, 2),      # eight, more clusters than have an SM per CTA; the last owner has two rows of three
])
def test_local_steps_rows_per_owner(dims, W, B, U):
    cfg = _small_cfg(inputs.SOFTMAX, dims, inputs.FP32, W, B, 3, 5, GAMMA3, lr=0.02)
    X, y, w0 = _problem(cfg)
    compare_with_oracle(cfg, X, y, w0, 6, TOL_FP32, forced=True, local_steps=U)
