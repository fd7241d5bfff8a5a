"""Work that users of the library have it do, as measurable cases.

A case is one call of the stand-alone gradient operation, or one training run the way the README shows it: create a
context over a dataset that is already on the device, run its rounds, read parameters and trace, release the context.
Shapes, batch sizes, worker counts, time laws and step sizes are those of the configurations in `inputs.config`, of
the parity tests and of `bench.py`'s options; the number of rounds is a configuration's own where such a run is short,
a part of it otherwise.

Runs in bf16 keep K fixed (`ABS_K_FIXED`, `bench.py --k-fixed`): with adaptive K a last-digit difference of an
uploaded loss can move a round's K by one, and from there on the two traces are different runs.  K is then set to the
regime a configuration spends its rounds in.  fp32 runs adapt K by Eq. 5.
"""
import math

import numpy as np
import torch

from paper_2301_08895_b200 import abs as gpu
from paper_2301_08895_b200 import inputs

LAWS = {
    "sexp": dict(kind=inputs.T_SHIFTED_EXP, shift=1.0, rate=1.0),
    "exp": dict(kind=inputs.T_EXP, rate=1.0),
    "slow": dict(kind=inputs.T_SHIFTED_EXP, shift=1.0, rate=1.0, slow_mod=10, slow_rem=9, slow_factor=5.0),
    "pareto": dict(kind=inputs.T_PARETO2, scale=1.0),
    "gamma": dict(kind=inputs.T_GAMMA, shift=0.0, rate=3.0, shape=3),
}
KINDS = {"lsq": inputs.LSQ, "softmax": inputs.SOFTMAX, "mlp": inputs.MLP, "cnn": inputs.CNN}


def _op(n, B, d, dtype, M, **kw):
    return dict(kind="op", n=n, B=B, d=d, dtype=dtype, M=M, **kw)


def _run(kind, dims, dtype, W, B, K0, S, rounds, lr, M, law, **kw):
    c = dict(kind=kind, dims=dims, dtype=dtype, W=W, B=B, K0=K0, S=S, rounds=rounds, lr=lr, M=M, law=law,
             adaptive=dtype == "fp32", U=1, clip=False, conv="", sa=0)
    c.update(kw)
    return c


def listed():
    return [
        # one stand-alone minibatch gradient of a few workers: the smallest call there is
        _op(8, 32, 64, "fp32", 8192, name="lsq_gradient"),
        # configuration 1: small least squares, the whole run
        _run("lsq", "64-1", "fp32", 8, 32, 2, 4, 200, 0.05, 8192, "sexp", name="lsq64"),
        # configuration 2: soft-max regression, the whole run
        _run("softmax", "784-10", "fp32", 16, 64, 4, 8, 1000, 0.1, 60000, "exp", clip=True, name="softmax784"),
        # configuration 2 with the paper's ten local steps per job
        _run("softmax", "784-10", "fp32", 16, 64, 4, 8, 100, 0.1, 60000, "exp", clip=True, U=10, name="softmax784_u10"),
        # a small fp32 network of odd widths, odd batch: none of the aligned paths applies
        _run("mlp", "300-123-57-7", "fp32", 13, 37, 3, 5, 200, 0.02, 20000, "pareto", name="mlp_ragged_fp32"),
        # configuration 3 with half of its workers per round, stragglers in the other half
        _run("mlp", "784-256-10", "bf16", 64, 128, 32, 8, 500, 0.1, 60000, "slow", clip=True, name="mlp784"),
        # configuration 3 with ten local steps per job: every worker trains a copy of the network
        _run("mlp", "784-256-10", "bf16", 64, 128, 32, 8, 40, 0.1, 60000, "slow", clip=True, U=10, name="mlp784_u10"),
        # configuration 4 where it spends nearly all of its rounds: every worker in every round
        _run("mlp", "3072-1024-512-10", "bf16", 128, 64, 128, 16, 300, 0.01, 50000, "pareto", name="mlp3072_all"),
        # configuration 4 with few arrivals of many staleness values per round (bench.py --k-fixed 16)
        _run("mlp", "3072-1024-512-10", "bf16", 128, 64, 16, 16, 400, 0.01, 50000, "pareto", name="mlp3072_k16"),
        # configuration 5 at its smallest worker count, half of the workers per round
        _run("lsq", "4096-1", "bf16", 256, 32, 128, 32, 500, 0.01, 262144, "exp", name="lsq4096_w256"),
        # configuration 5 at its largest worker count, all workers per round, the full dataset
        _run("lsq", "4096-1", "bf16", 1024, 32, 1024, 32, 500, 0.01, 1000000, "exp", name="lsq4096_w1024"),
        # configuration 6, the paper's own model class
        _run("cnn", "400-120-84-10", "bf16", 20, 32, 20, 8, 200, 0.003, 50000, "gamma", conv="32-32-3-5-6-16",
             name="cnn32"),
    ]


def _ints(text):
    return tuple(int(v) for v in text.split("-"))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["op", "lsq", "lsq", "softmax", "softmax_u", "mlp_fp32", "mlp", "mlp", "mlp_u", "cnn"])
    law, sa = rng.choice(sorted(LAWS)), int(rng.random() < 0.2)
    if family == "op":
        d = _log(rng, 16, 4096)
        return _op(_log(rng, 1, 256), _log(rng, 4, 256), d, rng.choice(["fp32", "bf16"]), 20000)
    W = _log(rng, 4, 128)
    K0 = max(1, int(W * rng.uniform(0.1, 1.0)))
    S = max(4, min(24, -(-W // K0) + rng.randrange(8)))
    if family == "lsq":
        dtype = rng.choice(["fp32", "bf16", "bf16"])
        d = _log(rng, 16, 4096)
        d = d if rng.random() < 0.3 else -(-d // 8) * 8
        W = _log(rng, 4, 1024)
        K0 = max(1, int(W * rng.uniform(0.1, 1.0)))
        S = max(4, min(32, -(-W // K0) + rng.randrange(8)))
        B = _log(rng, 8, 64)
        rounds = max(20, min(500, int((1.2e9 if d % 8 else 1.6e10) / (W * B * d))))
        lr = 0.3 / ((1 + math.sqrt(d / (K0 * B))) ** 2 * (1 + W / K0))      # stable with stale gradients
        return _run("lsq", "%d-1" % d, dtype, W, B, K0, S, rounds, lr, 40000, law, sa=sa)
    if family in ("softmax", "softmax_u"):
        W = min(W, 64)
        K0 = max(1, min(K0, W))
        U = rng.randrange(2, 11) if family == "softmax_u" else 1
        C, d = rng.choice([2, 5, 7, 10, 10, 16]), _log(rng, 32, 784)
        B = _log(rng, 16, 128)
        rounds = max(20, min(1000, int(2.5e9 / (W * B * d * U))))
        return _run("softmax", "%d-%d" % (d, C), "fp32", W, B, K0, S, rounds // (U if U > 1 else 1) + 20, 10.0 / d, 20000,
                    law, U=U, sa=sa)
    if family == "mlp_fp32":
        W = min(W, 24)
        K0 = max(1, min(K0, W))
        dims = [_log(rng, 32, 400)] + [_log(rng, 16, 160) for _ in range(rng.randrange(1, 3))] + [rng.randrange(3, 13)]
        return _run("mlp", "-".join(map(str, dims)), "fp32", W, _log(rng, 8, 64), K0, S, rng.randrange(60, 200), 5.0 / dims[0],
                    20000, law, sa=sa)
    if family in ("mlp", "mlp_u"):
        up8 = (lambda v: -(-v // 8) * 8) if rng.random() < 0.85 else (lambda v: v)
        U = rng.randrange(2, 11) if family == "mlp_u" else 1
        top = 3072 if U == 1 else 1024
        dims = [up8(_log(rng, 128, top))] + [up8(_log(rng, 64, 1024 if U == 1 else 384)) for _ in range(rng.randrange(1, 3))] + [10]
        B = _log(rng, 16, 128)
        work = W * B * U * sum(a * b for a, b in zip(dims, dims[1:]))       # multiply-adds of a pass over all workers
        aligned = all(v % 8 == 0 for v in dims[:-1])
        rounds = max(10, min(400, int((4e12 if aligned else 2.5e10) / work)))
        if not aligned:
            W = min(W, 32)
            K0 = min(K0, W)
        return _run("mlp", "-".join(map(str, dims)), "bf16", W, B, K0, S, rounds if U == 1 else min(40, rounds), 15.0 / dims[0],
                    20000, law, U=U, sa=sa)
    # the paper's model class on other image sizes and channel counts
    k = rng.choice([3, 5, 5])
    c1, c2 = rng.randrange(4, 9), rng.randrange(8, 17)
    side = rng.choice([v for v in range(14, 33) if (v - k + 1) % 2 == 0 and ((v - k + 1) // 2 - k + 1) % 2 == 0
                       and (v - k + 1) // 2 - k + 1 >= 2])
    ch = rng.choice([1, 3])
    feat = (((side - k + 1) // 2 - k + 1) // 2) ** 2 * c2
    W = min(W, 24)
    K0 = max(1, min(K0, W))
    return _run("cnn", "%d-%d-%d-10" % (feat, _log(rng, 48, 128), _log(rng, 32, 96)), rng.choice(["bf16", "bf16", "fp32"]), W,
                _log(rng, 8, 32), K0, S, 100, 0.003, 20000, law, conv="%d-%d-%d-%d-%d-%d" % (side, side, ch, k, c1, c2), sa=sa,
                adaptive=False)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    store = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    M, kind = case["M"], case["kind"]
    if kind == "op":
        d, n, B = case["d"], case["n"], case["B"]
        return dict(X=_randn(g, M, d).to(store), y=_randn(g, M), w=_randn(g, d).to(store),
                    idx=torch.randint(0, M, (n, B), generator=g, device="cuda", dtype=torch.int32),
                    g=torch.empty(d, device="cuda"), loss=torch.empty(n, device="cuda"),
                    scratch=torch.empty(n * d, device="cuda"))
    dims = _ints(case["dims"])
    conv = _ints(case["conv"]) if case["conv"] else None
    width = conv[0] * conv[1] * conv[2] if conv else dims[0]
    X = torch.empty(M, width, dtype=store, device="cuda")
    step = max(1, (1 << 26) // width)
    if kind == "lsq":                     # y = X w* + noise
        y = torch.empty(M, device="cuda")
        w_star = _randn(g, width)
        for r in range(0, M, step):
            x = _randn(g, min(step, M - r), width).to(store)
            X[r:r + step] = x
            y[r:r + step] = x.float() @ w_star + 0.1 * _randn(g, x.shape[0])
    else:                                 # Gaussian mixture, one mean per class
        means = _randn(g, dims[-1], width)
        y = torch.randint(0, dims[-1], (M,), generator=g, device="cuda", dtype=torch.int32)
        for r in range(0, M, step):
            lab = y[r:r + step].long()
            x = means[lab] + (2.0 if case["clip"] else 1.0) * _randn(g, lab.shape[0], width)
            X[r:r + step] = x.clamp_(0.0, 1.0) if case["clip"] else x
    w0 = np.zeros(inputs.n_params(KINDS[kind], dims, conv), dtype=np.float32)
    if kind in ("mlp", "cnn"):            # He-normal weights, zero biases
        blocks = [(a, a * b, b) for a, b in zip(dims, dims[1:])]
        if conv:
            _, _, c_in, k, c1, c2 = conv
            blocks = [(k * k * a, k * k * a * b, b) for a, b in ((c_in, c1), (c1, c2))] + blocks
        off = 0
        for fan_in, n_w, n_b in blocks:
            w0[off:off + n_w] = (_randn(g, n_w) * math.sqrt(2.0 / fan_in)).cpu().numpy()
            off += n_w + n_b
    args = (KINDS[kind], dims, X, y, w0, case["B"], case["lr"], case["W"], case["K0"], case["S"],
            inputs.TimeSpec(**LAWS[case["law"]]), seed, case["rounds"])
    kw = dict(dtype=gpu.BF16_FP32MASTER if case["dtype"] == "bf16" else gpu.FP32, local_steps=case["U"], conv=conv,
              k_mode=gpu.K_ADAPTIVE if case["adaptive"] else gpu.K_FIXED, sa_penalty=case["sa"])
    n_sel = case["rounds"] * (case["W"] if case["adaptive"] else case["K0"])
    return dict(args=args, kw=kw, rounds=case["rounds"], entries=(case["rounds"] * case["W"], n_sel))


def run(state):
    if "idx" in state:
        gpu.lsq_gradient(state["X"], state["y"], state["w"], state["idx"], state["g"], state["loss"], state["scratch"])
        return state["g"], state["loss"]
    ctx = gpu.Context(*state["args"], **state["kw"])
    ctx.run_rounds(state["rounds"])
    out = ctx.get_trace()
    out["params"] = ctx.get_params()
    ctx.close()
    for k in ("sel_id", "sel_tau", "sel_loss", "rst_id"):      # their lengths depend on the run: -1 behind the last entry
        short = state["entries"][k != "rst_id"] - len(out[k])
        if short:
            out[k] = np.pad(out[k], (0, short), constant_values=-1)
    return out


def work(case):
    """Multiply-adds of Eq. 2 for the rows of all rounds; bytes: the sampled rows, and per round the fp32 parameters
    read and written and one model version written.  Adaptive runs count W arrivals per round, which they reach within
    a few dozen rounds."""
    e = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "op":
        n, B, d = case["n"], case["B"], case["d"]
        return {"flops": 4.0 * n * B * d, "bytes": float(n * B * (d * e + 8) + d * (e + 4) + 4 * n)}
    dims = _ints(case["dims"])
    K = case["W"] if case["adaptive"] else case["K0"]
    rows = case["rounds"] * K * case["B"] * case["U"]
    width = dims[0]
    if case["kind"] == "lsq":
        per_row, n_par = 4.0 * dims[0], dims[0]
    else:
        per_layer = [2.0 * a * b for a, b in zip(dims, dims[1:])]
        per_row, n_par = 2 * sum(per_layer) + sum(per_layer[1:]), sum(a * b + b for a, b in zip(dims, dims[1:]))
    if case["conv"]:
        H, Wd, c_in, k, c1, c2 = _ints(case["conv"])
        h1, w1 = H - k + 1, Wd - k + 1
        h2, w2 = h1 // 2 - k + 1, w1 // 2 - k + 1
        f1, f2 = 2.0 * k * k * c_in * c1 * h1 * w1, 2.0 * k * k * c1 * c2 * h2 * w2
        per_row += per_layer[0] + f1 + 0.25 * f1 + f2 + 0.25 * f2 + 0.25 * f2   # deltas sit at the pooled maxima only
        n_par += k * k * c_in * c1 + c1 + k * k * c1 * c2 + c2
        width = H * Wd * c_in
    return {"flops": rows * per_row, "bytes": float(rows * (width * e + 4) + case["rounds"] * n_par * (8 + e))}


def tolerance(case):
    """Four times (or a little more) what the same run gives with its sums in another order: the FP32-FMA kernels in
    place of the tensor cores and of the bulk-copy pipeline, or binary64 for the fp32 cases.  In the convolutional
    network and in fp32 networks single ReLU and max-pool decisions fall differently and the runs drift apart."""
    if case["dtype"] == "bf16":
        return {"rel": {"cnn": 1e-2, "mlp": 5e-3}.get(case["kind"], 2e-3)}
    return {"rel": {"cnn": 1e-3, "mlp": 1e-4}.get(case["kind"], 1e-5)}
