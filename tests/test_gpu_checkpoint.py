"""Checkpoint / resume through the C ABI: a run that is saved after n rounds and continued in a
fresh context must be bit-identical (trace and parameters) to the uninterrupted run, which the
parity tests compare with the oracle."""
import numpy as np
import pytest

from paper_2301_08895_b200 import inputs
from helpers import gpu, to_device
from test_gpu_parity import _small_cfg, _problem, EXP, GAMMA3, PARETO

pytestmark = pytest.mark.gpu


def _ctx(cfg, X, y, w0, rounds, **kw):
    Xd, yd = to_device(cfg, X, y)
    return gpu.context_from_config(cfg, Xd, yd, w0, max_rounds=rounds, **kw), (Xd, yd)


@pytest.mark.parametrize("kind,dims,dtype,W,B,K0,S,time,kw", [
    (inputs.LSQ, (32, 1), inputs.FP32, 16, 8, 4, 6, EXP, {}),                                 # all rounds in one kernel
    (inputs.LSQ, (4096, 1), inputs.BF16, 64, 16, 8, 9, PARETO, {}),                           # bulk-copy pipeline
    (inputs.SOFTMAX, (40, 6), inputs.FP32, 12, 16, 3, 5, GAMMA3, {}),
    (inputs.MLP, (64, 128, 128, 10), inputs.BF16, 24, 32, 4, 7, EXP, {}),                     # tensor cores, two streams
    (inputs.MLP, (64, 128, 10), inputs.BF16, 8, 16, 3, 5, GAMMA3, {"local_steps": 3}),        # local steps
    (inputs.SOFTMAX, (24, 5), inputs.FP32, 10, 8, 2, 4, EXP, {"restart_rule": gpu.RESTART_EQ6}),
])
def test_resume_is_bit_identical(kind, dims, dtype, W, B, K0, S, time, kw):
    cfg = _small_cfg(kind, dims, dtype, W, B, K0, S, time, lr=0.02)
    X, y, w0 = _problem(cfg)
    n1, n2 = 13, 17
    a, keep_a = _ctx(cfg, X, y, w0, n1 + n2, **kw)
    a.run_rounds(n1 + n2)
    rows_a, params_a = gpu.trace_rows(a.get_trace()), a.get_params()
    a.close()

    b, keep_b = _ctx(cfg, X, y, w0, n1 + n2, **kw)
    b.run_rounds(n1)
    image = b.save_state()
    b.run_rounds(3)                      # the saving context may go on; the image is a copy
    b.close()

    c, keep_c = _ctx(cfg, X, y, w0, n1 + n2, **kw)
    c.restore_state(image)
    assert c.rounds_done()[0] == n1
    c.run_rounds(n2)
    rows_c, params_c = gpu.trace_rows(c.get_trace()), c.get_params()
    c.close()
    assert rows_c == rows_a
    assert np.array_equal(params_c.view(np.uint32), params_a.view(np.uint32))


HEADER_BLOCK1, HEADER_STATE, STATE_RB = 32, 152, 16       # byte offsets: size of the first region; state block; its row padding unit


def _region(W, rows_cap, RB, state, d_pad, esz, versions, shards):
    """(name, bytes) of the first region of an image in order, every piece on 256 bytes; shards: with the workers' shards
    and the tiles' real rows."""
    tiles = rows_cap // RB
    pieces = [("state", state), ("rounds", 32), ("c", 8 * W), ("version", 4 * W), ("job", 4 * W), ("next_dur", 8 * W), ("dur_job", 4 * W)]
    pieces += [("shard", 8 * W)] if shards else []
    for q in "01":
        pieces += [("sel" + q, 4 * W), ("tau" + q, 4 * W), ("row0" + q, 4 * W), ("idx" + q, 4 * rows_cap), ("slot" + q, 4 * tiles)]
        pieces += [("real" + q, 4 * tiles)] if shards else []
    pieces += [("loss", 4 * W), ("row_loss", 4 * rows_cap), ("master", 4 * d_pad), ("ring", esz * d_pad * versions)]
    out, off = {}, 0
    for name, n in pieces:
        out[name] = (off, n)
        off = -(-(off + n) // 256) * 256
    return out, off


def _older_image(image, cfg, plan, RB, shards, local_steps=1):
    """The image as a build with row padding unit RB, with or without shards (and without operand fragments), saved it."""
    W, B, S = cfg.W, cfg.batch, cfg.S
    esz = 2 if cfg.dtype == inputs.BF16 else 4
    block1 = int(image[HEADER_BLOCK1:HEADER_BLOCK1 + 8].view(np.uint64)[0])
    block2 = int(image[HEADER_BLOCK1 + 8:HEADER_BLOCK1 + 16].view(np.uint64)[0])
    d_pad = int(image[16:24].view(np.uint64)[0])
    header = len(image) - block1 - block2
    state = header - HEADER_STATE
    new, _ = _region(W, plan["rows_cap"], plan["row_block"], state, d_pad, esz, S + 1, True)
    rows_cap = -(-W * B // RB) * RB + min(W, S + 1) * RB
    if local_steps > 1:
        rows_cap = max(rows_cap, W * (-(-B // RB) * RB))
    old, size = _region(W, rows_cap, RB, state, d_pad, esz, S + 1, shards)
    region = np.full(size, 0xA5, np.uint8)                       # (what is not carried over must not be read)
    for name in ("state", "rounds", "c", "version", "job", "next_dur", "dur_job", "master", "ring"):
        (a, n), (b, _) = new[name], old[name]
        region[b:b + n] = image[header + a:header + a + n]
    head = image[:header].copy()
    for part in (head[HEADER_STATE:], region):
        part[STATE_RB:STATE_RB + 4].view(np.int32)[0] = RB
    head[HEADER_BLOCK1:HEADER_BLOCK1 + 8].view(np.uint64)[0] = size
    return np.concatenate([head, region, image[header + block1:]])


@pytest.mark.parametrize("kind,dims,dtype,W,B,RB,shards,kw", [
    (inputs.SOFTMAX, (40, 6), inputs.FP32, 12, 16, 64, False, {}),                      # row kernels; saved for 64-row tiles
    (inputs.SOFTMAX, (40, 6), inputs.FP32, 12, 16, 8, True, {}),
    (inputs.LSQ, (4096, 1), inputs.BF16, 64, 16, 16, False, {}),
    (inputs.MLP, (64, 128, 128, 10), inputs.BF16, 24, 32, 128, False, {}),
    (inputs.MLP, (64, 128, 10), inputs.BF16, 8, 16, 128, False, {"local_steps": 3}),
    (inputs.CNN, (64, 24, 10), inputs.BF16, 6, 16, 64, False, {}),                      # operand fragments made from the ring
    (inputs.CNN, (64, 24, 10), inputs.BF16, 6, 16, 128, True, {}),
])
def test_resume_from_an_image_of_another_layout(kind, dims, dtype, W, B, RB, shards, kw):
    """Images keep their pieces where the saving build's workspace had them; one of an earlier build (other row padding,
    no shards) continues bit-identically."""
    cfg = _small_cfg(kind, dims, dtype, W, B, 3, 5, GAMMA3, lr=0.01)
    if kind == inputs.CNN:
        cfg.conv, cfg.w0 = (14, 14, 3, 3, 4, 16), "he"
    X, y, w0 = _problem(cfg)
    a, keep_a = _ctx(cfg, X, y, w0, 20, **kw)
    a.run_rounds(9)
    image, plan = a.save_state(), a.plan()
    a.run_rounds(11)
    rows_a, params_a = gpu.trace_rows(a.get_trace()), a.get_params()
    a.close()
    old = _older_image(image, cfg, plan, RB, shards, kw.get("local_steps", 1))
    b, keep_b = _ctx(cfg, X, y, w0, 20, **kw)
    with pytest.raises(gpu.AbsError) as e:
        b.restore_state(old[:-1])
    assert e.value.code == gpu.EINVAL
    b.run_rounds(2)                      # (a context that has run already)
    b.restore_state(old)
    assert b.rounds_done()[0] == 9
    again = b.save_state()
    b.run_rounds(11)
    assert gpu.trace_rows(b.get_trace()) == rows_a
    assert np.array_equal(b.get_params().view(np.uint32), params_a.view(np.uint32))
    b.close()
    assert len(again) == len(image)


def test_restore_rejects_an_image_of_another_run():
    cfg = _small_cfg(inputs.LSQ, (32, 1), inputs.FP32, 16, 8, 4, 6, EXP, lr=0.02)
    X, y, w0 = _problem(cfg)
    a, keep = _ctx(cfg, X, y, w0, 20)
    a.run_rounds(5)
    image = a.save_state()
    a.close()
    import dataclasses
    other = dataclasses.replace(cfg, run_seed=cfg.run_seed + 1)
    b, keep_b = _ctx(other, X, y, w0, 20)
    with pytest.raises(gpu.AbsError) as e:
        b.restore_state(image)
    assert e.value.code == gpu.EINVAL
    with pytest.raises(gpu.AbsError) as e:
        b.restore_state(image[:100])
    assert e.value.code == gpu.EINVAL
    b.run_rounds(4)                      # the refused restore left the context usable
    assert b.rounds_done()[0] == 4
    b.close()
    c, keep_c = _ctx(cfg, X, y, w0, 30)  # other trace capacity
    with pytest.raises(gpu.AbsError) as e:
        c.restore_state(image)
    assert e.value.code == gpu.EINVAL
    c.close()
    # same sizes, other hyper-parameters: the image carries the model description and the modes
    for kw_other, cfg_other in (({}, dataclasses.replace(cfg, lr=0.03)),               # step size
                                ({"local_steps": 3}, cfg),                               # U (the upload block keeps its size)
                                ({"sa_penalty": 1}, cfg),                                # staleness-aware step size
                                ({"restart_rule": gpu.RESTART_NONE}, cfg),               # no forced restarts
                                ({"flags": gpu.FLAG_NO_PERSISTENT}, cfg)):               # another kernel path
        d, keep_d = _ctx(cfg_other, X, y, w0, 20, **kw_other)
        with pytest.raises(gpu.AbsError) as e:
            d.restore_state(image)
        assert e.value.code == gpu.EINVAL, kw_other
        d.close()
