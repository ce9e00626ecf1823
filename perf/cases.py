"""Workloads of the library as its users call it, for timing and for comparing outputs.

A case names an operation and its sizes.  The sizes are those of the benchmark and of the parity tests (univariate
16 x 512 with 1,000 kernels; 20 sensor channels of 5,000 and 50,000 steps with 10,000 kernels; the training pass of 32
examples; the regressor on 677 examples of 20,000 features) and generic ones around them: a single example, odd lengths,
few kernels, more channels than the paper's 20 sensors.

Operations
  hard           rocket_transform on device-resident fp32 samples
  f16            rocket_transform_f16, the same in binary16 arithmetic
  u8_host        rocket_transform_u8_host: raw 8-bit intensities in pinned host memory, features back in host memory
  train          one training pass: rocket_transform_soft, then rocket_transform_soft_backward with its argmax
  mini           MiniRocket.transform with fitted biases
  ridge_fit      rocket_ridge_fit on the features of a training set
  ridge_predict  rocket_ridge_predict on the features of a batch
"""
import functools
import math

import numpy as np
import torch

import paper_2301_08527_b200 as rk
from paper_2301_08527_b200 import binding

PARAM_SEED = 8527
LAMBDA, SHIFT, ALPHA = 10.0, 3.0, 1.0
PAPER = dict(C=20, L=50000, K=10000)


def listed():
    return [
        # a small univariate problem: launches and the host path weigh most
        dict(name="hard univariate", op="hard", N=16, C=1, L=512, K=1000),
        # an ordinary multivariate batch
        dict(name="hard batch", op="hard", N=64, C=20, L=5000, K=10000),
        # one second of the production line at once
        dict(name="hard paper scale", op="hard", N=60, **PAPER),
        # one example as it comes off the line: latency
        dict(name="hard streaming", op="hard", N=1, **PAPER),
        # more channels than the paper's sensors, an odd length, fewer kernels
        dict(name="hard many channels", op="hard", N=24, C=32, L=1751, K=2000),
        # reduced precision, a length that is no multiple of four
        dict(name="half precision", op="f16", N=8, C=20, L=10001, K=10000),
        # the sensors' bytes from host memory, end to end
        dict(name="bytes from the host", op="u8_host", N=60, **PAPER),
        # training the kernels: the paper-scale pass and a small minibatch of short, odd series
        dict(name="train paper scale", op="train", N=32, **PAPER),
        dict(name="train minibatch", op="train", N=10, C=6, L=1251, K=1000),
        # MINIROCKET on the same second of the line
        dict(name="minirocket", op="mini", N=60, C=20, L=50000, F=9996),
        # the regressor: fit on the paper's training set, predict for one batch (the smallest call)
        dict(name="ridge fit", op="ridge_fit", N=677, P=20000),
        dict(name="ridge predict", op="ridge_predict", N=60, P=20000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: Largest work of a drawn case (floating-point operations of one pass): what the listed cases of the same kind reach.
_MOST_FLOPS = {"hard": 1.5e12, "f16": 3e11, "u8_host": 1.5e12, "train": 2.5e12, "mini": 5e10, "ridge_fit": 1e10, "ridge_predict": 1e9}


def draw(rng):
    """One more case of the same ranges: batches from one example up, series of 64 to 100,000 steps, 1 to 32 channels,
    100 to 20,000 kernels, half of the sizes odd."""
    op = rng.choice(["hard", "hard", "hard", "f16", "u8_host", "train", "train", "mini", "ridge_fit", "ridge_predict"])
    while True:
        if op == "ridge_fit":
            case = dict(op=op, N=_log_int(rng, 24, 900), P=_log_int(rng, 200, 20000))
        elif op == "ridge_predict":
            case = dict(op=op, N=_log_int(rng, 1, 700), P=_log_int(rng, 200, 20000))
        else:
            case = dict(op=op, N=_log_int(rng, 1, 128), C=rng.choice([1, 2, 3, 6, 9, 12, 20, 20, 20, 20, 25, 32]), L=_log_int(rng, 64, 100000))
            if op == "f16":
                case["C"] = min(case["C"], 20)         # what the entry point accepts
            if op == "mini":
                case["F"] = 84 * _log_int(rng, 4, 119)
            else:
                case["K"] = _log_int(rng, 100, 20000)
        most = _MOST_FLOPS[op] / (8 if case.get("C", 1) > 20 else 1)
        if _rough_flops(case) <= most and case["N"] * case.get("C", 1) * case.get("L", case.get("P", 1)) <= 6.4e7:
            return case


def _rough_flops(case):
    if case["op"] == "ridge_fit":
        return float(case["N"]) ** 2 * case["P"]
    if case["op"] == "ridge_predict":
        return 2.0 * case["N"] * case["P"]
    if case["op"] == "mini":
        return 18.0 * case["N"] * case["L"] * min(case["F"], 84 * 32)
    channels = 0.3 + 0.45 * min(case["C"], 9) ** 0.9
    return 18.0 * channels * case["N"] * case["L"] * case["K"] * (3 if case["op"] == "train" else 1)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _series(N, C, L, g):
    """AR(1) noise (phi = 0.95) plus sparse positive spikes, unnormalised, [N, C, L] on the device."""
    phi, taps = 0.95, 512
    e = torch.randn((N, C, L + taps), generator=g, device="cuda")
    n = 1 << (L + 2 * taps - 1).bit_length()
    h = torch.fft.rfft(phi ** torch.arange(taps, device="cuda", dtype=torch.float32), n=n)
    out = torch.empty((N, C, L), device="cuda")
    for i in range(N):
        out[i] = torch.fft.irfft(torch.fft.rfft(e[i], n=n) * h, n=n)[:, taps:taps + L]
    spikes = torch.rand((N, C, L), generator=g, device="cuda") < 1e-3
    out += spikes * torch.empty_like(out).exponential_(1.0, generator=g)
    return out


def _normalised(x):
    return ((x - x.mean(-1, keepdim=True)) / x.std(-1, unbiased=False, keepdim=True).clamp_min(1e-6)).contiguous()


def prepare(case, seed):
    g = _generator(seed)
    op, N = case["op"], case["N"]
    state = {"op": op, "case": case}
    if op.startswith("ridge"):
        P = case["P"]
        # pooled features: shares of positive outputs in [0, 1] and maxima of order 1, in turn
        feat = torch.rand((N, P), generator=g, device="cuda")
        feat[:, 1::2] = 2.0 + 0.7 * torch.randn((N, P // 2), generator=g, device="cuda")
        w = torch.randn((P,), generator=g, device="cuda") / math.sqrt(P)
        state["feat"] = feat
        if op == "ridge_fit":
            state["y"] = (1.2 + (feat - feat.mean(0)) @ w + 0.1 * torch.randn((N,), generator=g, device="cuda")).contiguous()
        else:
            state["w"], state["b"] = w.contiguous(), torch.full((1,), 1.2, device="cuda")
        return state
    C, L = case["C"], case["L"]
    x = _series(N, C, L, g)
    if op == "mini":
        m = rk.MiniRocket.create(PARAM_SEED, C, L, case["F"])
        m.fit(_normalised(_series(1, C, L, _generator(17))).cpu().numpy())
        state["mini"], state["X"] = m, _normalised(x)
        return state
    params = rk.RocketParams.generate(PARAM_SEED, case["K"], C, L)
    state["params"] = params
    if op == "u8_host":
        gain = 12.0 + 28.0 * torch.rand((C, 1), generator=g, device="cuda")
        offset = 60.0 + 120.0 * torch.rand((C, 1), generator=g, device="cuda")
        v = (offset + gain * x * math.sqrt(1 - 0.95 ** 2)).round().clamp(0, 255).to(torch.uint8)
        state["X"] = v.cpu().pin_memory()
        state["mean"] = offset.reshape(-1).cpu().numpy()
        state["inv_std"] = (1.0 / gain).reshape(-1).cpu().numpy()
        state["feat"] = torch.empty((N, 2 * case["K"])).pin_memory()
        params.reserve(N, rk.PASS_HARD | rk.PASS_U8_INPUT)
        return state
    state["X"] = _normalised(x)
    if op == "train":
        state["dfeat"] = torch.randn((N, 2 * case["K"]), generator=g, device="cuda")
        params.reserve(N, rk.PASS_SOFT | rk.PASS_BACKWARD)
    else:
        params.reserve(N, rk.PASS_HARD)
    return state


def run(state):
    op = state["op"]
    if op == "hard":
        return rk.rocket_transform(state["params"], state["X"])
    if op == "f16":
        return rk.rocket_transform_f16(state["params"], state["X"])
    if op == "u8_host":
        return binding.rocket_transform_u8_host(state["params"], state["X"], state["mean"], state["inv_std"], state["feat"])
    if op == "train":
        feat, arg = rk.rocket_transform_soft(state["params"], state["X"], LAMBDA, SHIFT)
        dW, db = rk.rocket_transform_soft_backward(state["params"], state["X"], LAMBDA, SHIFT, state["dfeat"], arg)
        return {"feat": feat, "argmax": arg, "dW": dW, "db": db}
    if op == "mini":
        return state["mini"].transform(state["X"])
    if op == "ridge_fit":
        return rk.rocket_ridge_fit(state["feat"], state["y"], ALPHA)
    return rk.rocket_ridge_predict(state["feat"], state["w"], state["b"])


@functools.lru_cache(maxsize=None)
def _rocket_size(K, C, L):
    params = rk.RocketParams.generate(PARAM_SEED, K, C, L)
    flops, outputs = params.work()
    n_weights = params.n_weights
    params.close()
    return flops, outputs, n_weights


@functools.lru_cache(maxsize=None)
def _mini_size(C, L, F):
    """(conv outputs, channel sums, bias comparisons) of one example."""
    m = rk.MiniRocket.create(PARAM_SEED, C, L, F)
    a = m.host_arrays()
    m.close()
    outputs = np.where(a["padded"] != 0, L, L - 8 * a["dilation"]).astype(np.float64)
    return outputs.sum(), (outputs * (a["num_channels"] - 1)).sum(), (outputs * np.diff(a["feature_offset"])).sum()


def work(case):
    """Convolution work is counted as 2 * length * channels * outputs per kernel, twice that for the backward; the two
    pooling operations of an output come on top."""
    op, N = case["op"], case["N"]
    if op == "ridge_fit":
        P = case["P"]
        return {"bytes": 4.0 * (N * P + N + P), "flops": float(N) * N * P + N ** 3 / 3.0 + 4.0 * N * P}
    if op == "ridge_predict":
        return {"bytes": 4.0 * (N * case["P"] + case["P"] + N), "flops": 2.0 * N * case["P"]}
    C, L = case["C"], case["L"]
    if op == "mini":
        outputs, sums, compares = _mini_size(C, L, case["F"])
        return {"bytes": 4.0 * N * (C * L + case["F"]), "flops": N * (18.0 * outputs + sums + compares)}
    K = case["K"]
    flops, outputs, n_weights = _rocket_size(K, C, L)
    sample = 1 if op == "u8_host" else 4
    if op == "train":
        return {"bytes": 2.0 * N * C * L * 4 + 4.0 * N * K * (2 + 1 + 2 + 1) + 4.0 * (2 * n_weights + 2 * K),
                "flops": N * (3 * flops + 8 * outputs)}
    return {"bytes": float(N) * C * L * sample + 8.0 * N * K + 4.0 * n_weights, "flops": N * (flops + 2 * outputs)}


def tolerance(case):
    op = case["op"]
    if op == "f16":
        return "exact"           # every rounding of the half-precision transform is specified
    if op in ("hard", "u8_host", "mini"):
        # fp32 sums; an output within their rounding of zero (or of a bias) moves its share by 1 / outputs, and an
        # output range can be as short as a few dozen steps
        return {"rel": 1e-5, "max": 0.02}
    if op == "train":
        return {"rel": 1e-4, "max": 4e-3, "differ": 1e-3}
    return {"rel": 1e-5}
