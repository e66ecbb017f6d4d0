"""Timed cases: what a program that serves a quantized diffusion transformer has this library do.

Every case goes through the public entry points of ``paper_2509_24416_gb300.clq``.  Activations are N(0, 1) with a few
channels scaled (the outliers that the rotation is there for), FFN down-projection inputs are the GELU of that, weights
are N(0, 0.02^2), and the swap vector comes from a calibration batch of the same distribution, as a checkpoint holds it.
"""
import math

import torch

from paper_2509_24416_gb300 import clq

DTYPES = {"f16": torch.float16, "bf16": torch.bfloat16}
W_CODES = {"e4m3": None, "e2m3": clq.CLQ_CODES_E2M3, "packed": clq.CLQ_CODES_INT4_PACKED}

# One transformer block at 1024 px (batch 2 x 4096 tokens, hidden 1152): QKV, attention out, FFN up, FFN down.
BLOCK = ((1152, 3456), (1152, 1152), (1152, 4608), (4608, 1152))


def _layer(name, M, K, N, b, dtype, **more):
    case = dict(name=name, kind="layer", M=M, K=K, N=N, b=b, dtype=dtype, a_bits=4, w_bits=4, w_codes="e4m3", bias=True,
                gelu=False, outliers=0.01)
    case.update(more)
    return case


def listed():
    return [
        # One attention projection of a small latent (16 x 16 patches): a call that lasts microseconds, so launches and
        # the host's share of a call count.
        _layer("small_256", 256, 1152, 1152, 64, "f16"),
        # Ragged everywhere: a packed batch of 1357 tokens, K and N that no tile divides, no bias.
        _layer("ragged_1357", 1357, 1184, 1003, 32, "f16", bias=False),
        # The four layers of one block at 1024 px, one after the other, as a denoising step runs them.
        dict(name="block_8192", kind="block", M=8192, b=64, dtype="f16", outliers=0.01),
        # Video tokens (16 frames x 32 x 32 patches), FFN up.
        _layer("video_up_16384", 16384, 1152, 4608, 128, "bf16"),
        # Hidden size 3072 with 4096 image and 512 text tokens, FFN up.
        _layer("wide_up_4608", 4608, 3072, 12288, 128, "bf16", outliers=0.005),
        # The FFN down projection of the same block (input after GELU), weights in the compact resident layout.
        _layer("wide_down_4608", 4608, 12288, 3072, 128, "bf16", w_codes="e2m3", gelu=True, outliers=0.005),
        # The largest: many images in one batch through one wide layer.
        _layer("wide_up_65536", 65536, 3072, 12288, 64, "f16", outliers=0.005),
        # The 8-bit activation setting.
        _layer("w4a8_qkv_8192", 8192, 1152, 3456, 64, "f16", a_bits=8),
        # 8-bit activations and weights.
        _layer("w8a8_up_4096", 4096, 1152, 4608, 128, "bf16", a_bits=8, w_bits=8),
        # Asymmetric activation codes with the zero-point epilogue.
        _layer("asym_qkv_8192", 8192, 1152, 3456, 64, "f16", kind="asym"),
        # The single-launch form of a layer, with the workspace that a program keeps.
        _layer("fused_up_2048", 2048, 1152, 4608, 64, "f16", kind="fused"),
        # Offline: a layer made from its calibration batch and weights, and its storage form.
        dict(name="calibrate_3072", kind="calibrate", M=256, batch=4, K=3072, N=9216, b=128, dtype="bf16", outliers=0.005),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["layer"] * 7 + ["asym", "fused", "calibrate", "block"])
    dtype = rng.choice(["f16", "bf16"])
    if kind == "block":
        return dict(kind=kind, M=_between(rng, 512, 16384), b=rng.choice([32, 64, 128]), dtype=dtype, outliers=0.01)
    b = rng.choice([32, 64, 64, 128, 128, 256])
    bits = rng.choice([(4, 4)] * 4 + [(8, 4), (8, 8)]) if kind == "layer" else (4, 4)
    w_codes = rng.choice(["e4m3"] * 4 + ["e2m3", "packed"]) if kind == "layer" and bits == (4, 4) else "e4m3"
    step = max(b, 128 if w_codes == "e2m3" else 32)
    K = max(step, _between(rng, 256, 12288) // step * step)
    N = _between(rng, 64, 12288)
    if rng.random() < 0.75:
        N = max(32, N // 32 * 32)
    if kind == "calibrate":
        N = min(N, 3072 * 12288 // K // 32 * 32)
        return dict(kind=kind, M=_between(rng, 32, 512), batch=rng.choice([1, 2, 4, 8]), K=K, N=N, b=b, dtype=dtype, outliers=0.01)
    M = _between(rng, 16, 65536)
    most = 65536 * 3072 * 12288 // (12 if bits[1] == 8 else 4)  # 8-bit weights cost four products
    while M * K * N > most or M * N > 65536 * 12288 // 2:
        M = M // 2
    case = _layer("", M, K, N, b, dtype, kind=kind, a_bits=bits[0], w_bits=bits[1], w_codes=w_codes, bias=rng.random() < 0.75,
                  gelu=rng.random() < 0.25)
    del case["name"]
    return case


# ------------------------------------------------------------------- inputs --
def _activations(g, shape, scale, dtype, gelu):
    x = torch.randn(shape, generator=g, device="cuda") * scale
    if gelu:
        x = torch.nn.functional.gelu(x)
    return x.to(dtype)


def _swap_vector(calib):
    """Channels ranked by max over tokens of |mean over the batch| (fp32, summed in order), the upper half first."""
    s = torch.zeros(calib.shape[1:], device=calib.device)
    for part in calib:
        s = s + part.float()
    scores = (s / calib.shape[0]).abs().amax(0)
    K = scores.numel()
    order = torch.sort(scores, descending=True, stable=True).indices
    high = torch.zeros(K, dtype=torch.bool, device=calib.device)
    high[order[:K // 2]] = True
    at = torch.arange(K, device=calib.device)
    return scores, torch.cat([at[high], at[~high]]).to(torch.int32)


def _inputs(case, K, N, M, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dtype = DTYPES[case["dtype"]]
    scale = torch.ones(K, device="cuda")
    count = max(1, round(case["outliers"] * K))
    at = torch.randperm(K, generator=g, device="cuda")[:count]
    scale[at] = 20 + 40 * torch.rand(count, generator=g, device="cuda")
    gelu = case.get("gelu", False) or (case["kind"] == "block" and K == 4608)
    calib = _activations(g, (case.get("batch", 4), case["M"] if case["kind"] == "calibrate" else 256, K), scale, dtype, gelu)
    W = (0.02 * torch.randn((N, K), generator=g, device="cuda")).to(dtype)
    bias = (0.01 * torch.randn(N, generator=g, device="cuda")).to(dtype) if case.get("bias", True) else None
    X = _activations(g, (M, K), scale, dtype, gelu) if case["kind"] != "calibrate" else None
    return X, W, bias, calib


def _shapes(case):
    return BLOCK if case["kind"] == "block" else ((case["K"], case["N"]),)


def _each(case, seed):
    for i, (K, N) in enumerate(_shapes(case)):
        yield _inputs(case, K, N, case["M"], seed * 16 + i)


def prepare(case, seed):
    kind = case["kind"]
    state = dict(kind=kind, case=case, layers=[])
    for X, W, bias, calib in _each(case, seed):
        if kind == "calibrate":
            state.update(W=W, calib=calib, bias=bias)
            break
        perm = _swap_vector(calib)[1]
        layer = clq.PreparedLinear.from_weight(W, perm, case["b"], bias=bias, a_bits=case.get("a_bits", 4),
                                               w_bits=case.get("w_bits", 4), w_codes=W_CODES[case.get("w_codes", "e4m3")])
        state["layers"].append((layer, X))
        if kind == "asym":
            state["wsum"] = clq.weight_code_sums(layer.We, layer.K)
        if kind == "fused":
            state["workspace"] = clq.fused_workspace(X.shape[0], layer.K, X.device)
    return state


def run(state):
    kind = state["kind"]
    if kind == "calibrate":
        layer, info = clq.PreparedLinear.calibrate(state["W"], state["calib"], state["case"]["b"], bias=state["bias"])
        d = layer.state_dict()
        return dict(scores=info["scores"], perm=d["perm"], Wq=d["Wq"], s_w=d["s_w"])
    if kind == "asym":
        layer, X = state["layers"][0]
        Xq, delta, lo = clq.rotate_quant_act_asym(X, layer.perm, layer.b)
        return clq.linear_asym(Xq, delta, lo, layer.We, layer.s_w, state["wsum"], layer.b, layer.K, bias=layer.bias,
                               out_dtype=X.dtype)
    if kind == "fused":
        layer, X = state["layers"][0]
        return layer(X, fused=True, workspace=state["workspace"])
    return [layer(X) for layer, X in state["layers"]]


# --------------------------------------------------------- what it comes to --
def work(case):
    M, total, flops = case["M"], 0, 0
    for K, N in _shapes(case):
        if case["kind"] == "calibrate":  # calibration batch and weights in; packed codes, scales, scores and swap vector out
            total += case["batch"] * M * K * 2 + N * K * 2 + N * K // 2 + 4 * N + 8 * K
            flops += N * K * int(math.log2(case["b"])) + case["batch"] * M * K
            continue
        w = {"e4m3": 1.0, "e2m3": 0.75, "packed": 0.5}[case.get("w_codes", "e4m3")] * (2 if case.get("w_bits", 4) == 8 else 1)
        total += M * K * 2 + int(N * K * w) + M * N * 2 + 4 * (N + K)
        flops += 2 * M * K * N + M * K * int(math.log2(case["b"]))
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Two correct implementations round the rotation, the scale and the ratio x / s differently in the last bits of 32,
    # so a few codes that lie at a tie come out one apart; outputs are rounded once to 16 bits.  Against exact() the listed cases and
    # fourteen drawn ones showed at most 9.2e-4 (f16) and 1.7e-3 (bf16), and 0.12 in the output a flipped code moves most.
    if case["kind"] == "calibrate":
        return {"rel": 1e-6, "differ": 1e-4}
    return {"rel": 4e-3, "max": 0.45} if case["dtype"] == "f16" else {"rel": 7e-3, "max": 0.45}


def _rotated(x, perm, b):
    i = torch.arange(b, device=x.device)
    ones = i[:, None] & i[None, :]
    sign = torch.zeros_like(ones)
    for k in range(8):
        sign ^= (ones >> k) & 1
    H = (1 - 2 * sign).double()
    x = x.double()[:, perm.long()]
    return (x.reshape(-1, b) @ H).reshape(x.shape)


def _symmetric(x, qmax):
    s = x.abs().amax(1, keepdim=True) / qmax
    q = torch.round(x / torch.where(s > 0, s, torch.ones_like(s))).clamp(-qmax, qmax)
    return q, s


def exact(case, seed):
    outs = []
    for X, W, bias, calib in _each(case, seed):
        scores, perm = _swap_vector(calib)
        b = case["b"]
        qw, sw = _symmetric(_rotated(W, perm, b), 127 if case.get("w_bits", 4) == 8 else 7)
        if case["kind"] == "calibrate":
            return dict(scores=scores.double(), perm=None, Wq=None, s_w=sw[:, 0])
        wd = (qw * (sw / b)).t().contiguous()
        Y = torch.empty((X.shape[0], W.shape[0]), dtype=torch.float64, device=X.device)
        for at in range(0, X.shape[0], 4096):
            x = _rotated(X[at:at + 4096], perm, b)
            if case["kind"] == "asym":
                lo, hi = x.amin(1, keepdim=True), x.amax(1, keepdim=True)
                span = torch.where(hi > lo, hi - lo, torch.ones_like(lo))
                xd = torch.round((x - lo) / span * 15) * ((hi - lo) / 15) + lo
            else:
                q, s = _symmetric(x, 127 if case.get("a_bits", 4) == 8 else 7)
                xd = q * s
            Y[at:at + 4096] = xd @ wd
        if bias is not None:
            Y += bias.double()
        outs.append(Y)
    return outs[0] if case["kind"] in ("asym", "fused") else outs
