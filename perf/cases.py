"""The work that users of this library have it do, as timed cases.

A case is one pass through the public entry points of paper_1901_03040_b200.qesgd on torch tensors.
Kinds:
  round      K workers copy the server's parameter, run one local epoch each, encode their deltas,
             the server decodes, averages and applies (Algorithm 3 on logistic regression)
  epoch      the local epoch of K workers alone
  qstep      one inner iteration of Algorithm 2: gradient step, requantise, running sum
  push       K workers push quantised minibatch gradients (the QSGD baseline): gradient of each,
             one encode without anchor, the server's axpy
  codec      encode of K workers' parameters against the anchor, then decode-average-apply
  aggregate  the server's half alone: decode-average-apply of K streams
  roundtrip  one vector encoded without anchor and decoded again
  requantize the quantisation of an inner iterate with write-back and running sum

Sizes are those of the benchmark configurations and tests (logistic regression with 65 536 features,
11 689 512 and 25 557 032 parameters, vectors of 2^24 to 2^28) or generic ones between them.
"""
import math

import torch

from paper_1901_03040_b200 import qesgd, synthetic

LEVELS = {2: 1, 4: 7, 8: 127}
MODES = {"norm": qesgd.SCALE_NORM, "max": qesgd.SCALE_MAX, "fixed": qesgd.SCALE_FIXED}
LR = 0.1
SEED = 7            # of the quantiser's draws


def listed():
    return [
        # a small problem, as in a first experiment: latency and launches count
        dict(name="round_small", kind="round", K=4, n_local=128, d=4096, batch=32, bits=8, bucket=512, mode="norm"),
        # the end-to-end configuration: 8192 samples of 65 536 features over four workers
        dict(name="round_logistic", kind="round", K=4, n_local=2048, d=65536, batch=64, bits=8, bucket=512, mode="norm"),
        # local epochs of eight workers on a middling number of features, ragged last minibatch
        dict(name="epoch_middling", kind="epoch", K=8, n_local=1010, d=10000, batch=50),
        # more features than the benchmark's
        dict(name="epoch_wide", kind="epoch", K=4, n_local=512, d=131072, batch=64),
        # the inner iteration of Algorithm 2 on a minibatch far larger than any cache
        dict(name="qstep_large", kind="qstep", m=64, d=1 << 22, bits=8, bucket=512, mode="norm"),
        # the baseline that quantises gradients: four workers, minibatches of 64
        dict(name="push_gradients", kind="push", K=4, m=64, d=65536, bits=8, bucket=512, mode="norm"),
        # ResNet-50-sized parameter, 16 workers, 2-bit codes: the default benchmark round
        dict(name="codec_resnet50", kind="codec", K=16, d=25_557_032, bits=2, bucket=256, mode="norm", pad=True,
             heavy=False),
        # workers' parameters as rows of one contiguous [K, d] tensor with an odd d, largest-magnitude scale
        dict(name="codec_odd_rows", kind="codec", K=5, d=1_000_003, bits=4, bucket=128, mode="max", pad=False,
             heavy=False),
        # heavy-tailed deltas, wide buckets, the largest vectors
        dict(name="codec_sweep", kind="codec", K=8, d=1 << 28, bits=4, bucket=4096, mode="norm", pad=True, heavy=True),
        # the server of eight workers with a ResNet-18-sized parameter
        dict(name="aggregate_resnet18", kind="aggregate", K=8, d=11_689_512, bits=4, bucket=512, mode="norm"),
        # the quantiser on one delta vector, and back
        dict(name="roundtrip_8bit", kind="roundtrip", d=1 << 24, bits=8, bucket=512, mode="norm"),
        # per-step quantisation of a network's parameter with a caller-given grid
        dict(name="requantize_large", kind="requantize", d=1 << 26, bits=8, bucket=512, mode="fixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round", "epoch", "qstep", "push", "codec", "aggregate", "roundtrip", "requantize"])
    bits = rng.choice([2, 4, 8])
    bucket = rng.choice([64, 128, 256, 512, 1024, 4096])
    mode = rng.choice(["norm", "norm", "max"])
    c = dict(kind=kind)
    if kind in ("round", "epoch"):
        K, d = rng.randint(1, 8), _log_int(rng, 100, 140_000)
        if rng.random() < 0.75:
            d = (d + 3) // 4 * 4                       # most feature counts are padded to a multiple of 4
        batch = rng.choice([16, 32, 50, 64, 100, 128])
        # at most the data of the end-to-end configuration
        n_local = min(_log_int(rng, batch, 2048), max(batch, (1 << 29) // (K * d)))
        c.update(K=K, n_local=n_local, d=d, batch=batch)
        if kind == "round":
            c.update(bits=bits, bucket=bucket, mode=mode)
    elif kind == "qstep":
        c.update(m=rng.choice([16, 33, 64, 128]), d=_log_int(rng, 4096, 1 << 21) // 4 * 4, bits=bits,
                 bucket=min(bucket, 1024), mode=mode)
    elif kind == "push":
        c.update(K=rng.randint(1, 8), m=rng.choice([16, 33, 64, 100, 256]), d=_log_int(rng, 1000, 300_000),
                 bits=bits, bucket=bucket, mode=mode)
    elif kind == "codec":
        K = rng.choice([1, 2, 3, 4, 5, 8, 10, 16, 32])
        c.update(K=K, d=_log_int(rng, 10_000, (1 << 29) // K), bits=bits, bucket=bucket, mode=mode,
                 pad=rng.random() < 0.75, heavy=rng.random() < 0.5)
    elif kind == "aggregate":
        K = rng.choice([1, 2, 3, 4, 5, 8, 10, 16, 32])
        c.update(K=K, d=_log_int(rng, 10_000, (1 << 28) // K), bits=bits, bucket=bucket, mode=mode)
    elif kind == "roundtrip":
        c.update(d=_log_int(rng, 10_000, 1 << 27), bits=bits, bucket=bucket, mode=mode)
    else:
        c.update(d=_log_int(rng, 10_000, 1 << 27), bits=bits, bucket=bucket, mode=rng.choice(["norm", "fixed"]))
    return c


# ----------------------------------------------------------------- inputs ----
def _normal(shape, sigma, seed, stream, heavy=False):
    return synthetic.device_normal_f32(shape, sigma, seed * 64 + stream, "cuda", 0.01 if heavy else 0.0)


def _logistic(rows, d, seed):
    """x ~ N(0, 1/d), y = sign(x . w*) with 5 % of the labels flipped, on the device."""
    X = _normal((rows, d), 1.0 / math.sqrt(d), seed, 1)
    y = torch.where(X @ _normal((d,), 1.0, seed, 2) >= 0.0, 1.0, -1.0)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 64 + 3)
    return X, torch.where(torch.rand(rows, device="cuda", generator=g) < 0.05, -y, y)


def _streams(st, K, d, bucket, bits):
    st["codes"], st["scales"] = qesgd.alloc_stream_buffers(K, d, bucket, bits, "cuda")


def prepare(case, seed):
    st = dict(case)
    kind, d = case["kind"], case["d"]
    st["ctx"] = qesgd.Context(0, None)
    st["epoch"] = 0
    if kind not in ("epoch",):
        st["s"], st["mode"] = LEVELS[case["bits"]], MODES[case["mode"]]
        codec = (d, case["bucket"], case["bits"])
    if kind in ("round", "epoch"):
        K = case["K"]
        st["X"], st["y"] = _logistic(K * case["n_local"], d, seed)
        st["param"] = _normal((d,), synthetic.ANCHOR_SIGMA, seed, 4)
        st["u"] = st["param"].repeat(K, 1)
        if kind == "round":
            _streams(st, K, *codec)
    elif kind == "qstep":
        st["X"], st["y"] = _logistic(case["m"], d, seed)
        st["anchor"] = _normal((d,), synthetic.ANCHOR_SIGMA, seed, 4)
        st["u"] = st["anchor"] + _normal((d,), 1e-3, seed, 5)
        st["zsum"] = _normal((d,), 0.05, seed, 6)       # of the iterations before
        _streams(st, 1, *codec)
    elif kind == "push":
        K = case["K"]
        X, y = _logistic(K * case["m"], d, seed)
        st["batches"] = [(X[k * case["m"]:(k + 1) * case["m"]], y[k * case["m"]:(k + 1) * case["m"]]) for k in range(K)]
        st["param"] = _normal((d,), synthetic.ANCHOR_SIGMA, seed, 4)
        st["stride"] = (d + 7) // 8 * 8
        st["grad"] = torch.zeros((K, st["stride"]), device="cuda")
        _streams(st, K, *codec)
    elif kind in ("codec", "aggregate"):
        K = case["K"]
        pad, heavy = case.get("pad", True), case.get("heavy", False)
        st["stride"] = (d + 7) // 8 * 8 if pad else d
        st["param"] = _normal((d,), synthetic.ANCHOR_SIGMA, seed, 4)
        st["local"] = _normal((K, st["stride"]), 1e-3, seed, 5, heavy)
        st["local"][:, :d] += st["param"]
        _streams(st, K, *codec)
        if kind == "aggregate":             # the streams have arrived: only they stay
            _encode(st, st["param"])
            torch.cuda.synchronize()
            del st["local"]
    elif kind == "roundtrip":
        st["local"] = _normal((d,), 1e-3, seed, 5)
        st["out"] = torch.empty(d, device="cuda")
        _streams(st, 1, *codec)
    else:                                   # requantize
        st["anchor"] = _normal((d,), synthetic.ANCHOR_SIGMA, seed, 4)
        st["u"] = st["anchor"] + _normal((d,), 1e-3, seed, 5)
        st["zsum"] = torch.zeros(d, device="cuda")
        _streams(st, 1, *codec)
    return st


# ------------------------------------------------------------------ passes ---
def _epoch(st):
    st["ctx"].qesgd_lr_local_epoch_batch(st["X"], st["y"], st["n_local"], st["d"], st["K"], st["batch"], LR,
                                         st["u"], st["d"])


def _encode(st, anchor):
    c, s = st["codes"], st["scales"]
    st["ctx"].qesgd_encode_batch(st["local"], st["stride"], anchor, st["d"], st["K"], st["bucket"], st["s"],
                                 st["bits"], st["mode"], SEED, 0, st["epoch"], c, c.stride(0), s, s.stride(0))


def _apply(st):
    c, s = st["codes"], st["scales"]
    st["ctx"].qesgd_decode_average_apply(st["param"], st["d"], st["K"], c, c.stride(0), s, s.stride(0),
                                         st["bucket"], st["s"], st["bits"])


def run(st):
    kind, ctx, d = st["kind"], st["ctx"], st["d"]
    st["epoch"] += 1
    if kind == "epoch":
        _epoch(st)
        return st["u"]
    if kind == "round":
        st["u"].copy_(st["param"].expand(st["K"], d))
        _epoch(st)
        st["local"], st["stride"] = st["u"], d
        _encode(st, st["param"])
        _apply(st)
        return st["u"], st["codes"], st["scales"], st["param"]
    if kind == "qstep":
        ctx.qesgd_lr_qesgd_step(st["X"], st["y"], st["m"], d, LR, st["u"], st["anchor"], st["bucket"], st["s"],
                                st["bits"], st["mode"], SEED, 0, st["epoch"], st["zsum"], st["codes"], st["scales"])
        return st["u"], st["zsum"], st["codes"], st["scales"]
    if kind == "push":
        for k, (X, y) in enumerate(st["batches"]):
            ctx.qesgd_lr_gradient(X, y, st["m"], d, st["param"], st["grad"][k])
        st["local"] = st["grad"]
        _encode(st, None)
        c, s = st["codes"], st["scales"]
        ctx.qesgd_decode_average_axpy(st["param"], d, st["K"], c, c.stride(0), s, s.stride(0), st["bucket"],
                                      st["s"], st["bits"], -LR)
        return st["grad"], c, s, st["param"]
    if kind == "codec":
        _encode(st, st["param"])
        _apply(st)
        return st["codes"], st["scales"], st["param"]
    if kind == "aggregate":
        _apply(st)
        return st["param"]
    if kind == "roundtrip":
        ctx.qesgd_encode(st["local"], None, d, st["bucket"], st["s"], st["bits"], st["mode"], SEED, 0, st["epoch"],
                         st["codes"], st["scales"])
        ctx.qesgd_decode(st["codes"], st["scales"], d, st["bucket"], st["s"], st["bits"], st["out"])
        return st["codes"], st["scales"], st["out"]
    ctx.qesgd_requantize(st["u"], st["anchor"], d, st["bucket"], st["s"], st["bits"], st["mode"], SEED, 0,
                         st["epoch"], st["zsum"], st["codes"], st["scales"], fixed_delta=4e-3 / st["s"])
    return st["u"], st["zsum"], st["codes"], st["scales"]


def work(case):
    """Each input read once and each output written once; two operations per multiply-add of the
    logistic passes (the codec's integer work is not counted)."""
    kind, d = case["kind"], case["d"]
    stream = case["bits"] / 8.0 + 4.0 / case["bucket"] if "bits" in case else 0.0    # bytes per element of a stream
    if kind in ("round", "epoch"):
        K, rows = case["K"], case["K"] * case["n_local"]
        b, f = 4.0 * rows * d + 4.0 * rows + 8.0 * K * d, 4.0 * rows * d
        if kind == "round":
            b += 4.0 * d + K * d * (4.0 + stream) + 4.0 * d + K * d * stream + 8.0 * d
        return {"bytes": b, "flops": f}
    if kind == "qstep":
        return {"bytes": 4.0 * case["m"] * d + d * (12.0 + 8.0 + stream), "flops": 4.0 * case["m"] * d}
    if kind == "push":
        K, m = case["K"], case["m"]
        return {"bytes": K * (4.0 * m * d + 8.0 * d) + K * d * (4.0 + 2.0 * stream) + 8.0 * d, "flops": 4.0 * K * m * d}
    if kind == "codec":
        K = case["K"]
        return {"bytes": d * (K * (4.0 + stream) + 4.0) + d * (K * stream + 8.0), "flops": 0.0}
    if kind == "aggregate":
        return {"bytes": d * (case["K"] * stream + 8.0), "flops": 0.0}
    if kind == "roundtrip":
        return {"bytes": d * (8.0 + 2.0 * stream), "flops": 0.0}
    return {"bytes": d * (20.0 + stream), "flops": 0.0}


def tolerance(case):
    """Four times what was seen against the same passes with their sums in 64 bits.  Codes, scales and
    everything decoded from them one by one are exact by contract.  An average over workers is a sum
    of fp32 terms in one order of several; logistic steps are fp32 dot products of d terms.  Behind
    them a delta u - w differs by the spacing of fp32 numbers at w, and with it the scale and the few
    codes whose draw lies on the boundary (three codes are allowed for the smallest vectors)."""
    kind, d = case["kind"], case["d"]
    if kind in ("roundtrip", "requantize"):
        return "exact"
    if kind in ("codec", "aggregate"):
        return {"rel": 1e-7, "max": 1.2e-6}
    if kind == "epoch":
        return {"rel": 6e-7, "max": 3e-6}
    few = 3.0 / (case.get("K", 1) * d * case["bits"] / 8.0)          # three bytes of the code streams
    if kind == "push":
        return {"rel": 5e-7, "max": 2e-4, "differ": 2e-5 + few}
    if kind == "qstep":
        return {"rel": 1e-6, "max": 0.999, "differ": 1e-6 + few}
    return {"rel": 1.5e-4, "max": 0.015, "differ": 7e-4 + few}
