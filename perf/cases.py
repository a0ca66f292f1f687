"""What users of this library have it do, as cases that can be timed and compared: weights expanded when a model is loaded
or swapped in, single linear layers, two-layer MLPs of the ensemble's predictors from one token to a full prefill,
convolutions and convolution stages, and layers on asymmetric activations.

A case is a dict of plain values.  Shapes and distributions are those of the configurations in ``synth.py`` (ConvNet, BERT
and LLM shaped layers) or generic; the online cases start from the fp32 activations a program holds and include their
quantization.
"""
from __future__ import annotations

import math

import torch

from paper_2311_15806_b200 import binding as B

ACTS = {"identity": B.ACT_IDENTITY, "relu": B.ACT_RELU, "silu": B.ACT_SILU, "gelu": B.ACT_GELU}

# Quantization settings of one layer: weight bits, orders K, channels per group g, kept fraction gamma, predictors M,
# distribution of the weights.
INT8 = {"bits": 8, "K": 2, "g": 8, "gamma": 1.0, "M": 1, "w": "normal_rowmult"}
INT4_BERT = {"bits": 4, "K": 4, "g": 8, "gamma": 0.5, "M": 2, "w": "normal_outliers"}
INT4_LLM = {"bits": 4, "K": 4, "g": 8, "gamma": 0.5, "M": 2, "w": "normal_rowmult"}
INT4_CONV = {"bits": 4, "K": 3, "g": 8, "gamma": 0.25, "M": 1, "w": "student_t"}
TERNARY = {"bits": 2, "K": 8, "g": 16, "gamma": 0.25, "M": 4, "w": "student_t"}


def listed() -> list[dict]:
    return [
        # One small int8 layer on a small batch: the call whose time is launches and latency.
        {"name": "linear_int8_t64", "op": "linear", "T": 64, "O": 256, "I": 256, "x": "normal", **INT8},
        # Decode: the two projections of an LLM-shaped MLP on one new token, the predictors of the ensemble added at the end.
        {"name": "mlp_decode_t1", "op": "mlp", "T": 1, "O": 4096, "I": 4096, "H": 11008, "x": "chan_outliers", "act": "silu",
         "int8_copy": False, **INT4_LLM},
        # Decode for 13 sequences at a time.
        {"name": "mlp_decode_t13", "op": "mlp", "T": 13, "O": 4096, "I": 4096, "H": 11008, "x": "chan_outliers", "act": "silu",
         "int8_copy": False, **INT4_LLM},
        # A large decode batch or a short prompt; not a multiple of any tile.
        {"name": "mlp_batch_t100", "op": "mlp", "T": 100, "O": 4096, "I": 4096, "H": 11008, "x": "chan_outliers", "act": "silu",
         "int8_copy": False, **INT4_LLM},
        # Prefill of a long prompt, on a layer that keeps the int8 copy meant for many tokens at a time.
        {"name": "mlp_prefill_t4096", "op": "mlp", "T": 4096, "O": 4096, "I": 4096, "H": 11008, "x": "chan_outliers",
         "act": "silu", "int8_copy": True, **INT4_LLM},
        # BERT-base-shaped feed-forward network on 32 sequences of 128 tokens.
        {"name": "ffn_t4096", "op": "mlp", "T": 4096, "O": 768, "I": 768, "H": 3072, "x": "normal", "act": "gelu",
         "int8_copy": False, **INT4_BERT},
        # An inner ternary layer of high order: every predictor has an input of its own.
        {"name": "linear_ternary_t8192", "op": "linear", "T": 8192, "O": 8192, "I": 8192, "x": "normal", **TERNARY},
        # A 3 x 3 convolution of a ConvNet's early stage, fp32 output.
        {"name": "conv_256_56x56", "op": "conv", "N": 32, "H": 56, "C": 256, "O": 256, "k": 3, "stride": 1, "x": "relu",
         **INT4_CONV},
        # Two inner convolutions of a late stage, the first one halving the image: int8 from layer to layer.
        {"name": "conv_stage_14x14", "op": "conv_stage", "N": 32, "H": 28, "C": 256, "O": 512, "k": 3, "stride": 2,
         "x": "relu", **INT4_CONV, "M": 2},
        # Asymmetric 8-bit activations (zero point) on a ragged batch of sequences.
        {"name": "asym_ffn_t709", "op": "asym", "T": 709, "O": 3072, "I": 768, "x": "relu", **INT4_BERT},
        # Loading (or swapping) the weights of an LLM-shaped MLP: both projections.
        {"name": "expand_mlp", "op": "expand", "O": 11008, "I": 4096, "pair": True, "int8_copy": False, **INT4_LLM},
        # The same for a ternary layer of eight orders.
        {"name": "expand_ternary", "op": "expand", "O": 8192, "I": 8192, "pair": False, "int8_copy": False, **TERNARY},
    ]


def _log(rng, lo: int, hi: int, step: int = 1) -> int:
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def _layer(rng) -> dict:
    bits = rng.choice([8, 4, 4, 4, 2, 6, 3])
    K = rng.randint(1, 8 if bits == 2 else 4)
    return {"bits": bits, "K": K, "g": 16 if bits == 2 else rng.choice([8, 16]), "gamma": rng.choice([0.25, 0.5, 0.75, 1.0]),
            "M": rng.randint(1, min(4, K)), "w": rng.choice(["normal_rowmult", "student_t", "normal_outliers"])}


def draw(rng) -> dict:
    # Widths are multiples of 16 (half of them of 128), from narrow heads to the widest LLM projections; token counts
    # from one to a long prefill, any number.
    def width(lo=128, hi=11008):
        return _log(rng, lo, hi, rng.choice([16, 128]))

    while True:
        op = rng.choice(["linear", "mlp", "mlp", "conv", "conv_stage", "lowered", "asym", "expand", "expand"])
        c = {"op": op, **_layer(rng)}
        if op == "linear":
            c.update(T=_log(rng, 1, 8192), O=width(), I=width(), x=rng.choice(["normal", "chan_outliers"]))
        elif op == "mlp":
            d = width(256, 4096)
            c.update(T=_log(rng, 1, 8192), O=d, I=d, H=width(512), x=rng.choice(["normal", "chan_outliers"]),
                     act=rng.choice(["relu", "silu", "gelu"]), int8_copy=rng.random() < 0.3)
        elif op in ("conv", "conv_stage"):
            c.update(N=rng.randint(1, 32), H=rng.choice([7, 14, 15, 28, 33, 56]), C=rng.choice([128, 256, 512]),
                     O=_log(rng, 64, 512, 16), k=rng.choice([1, 3, 3]), stride=rng.choice([1, 2]), x="relu")
            if op == "conv":
                c["M"] = 1
            else:
                c["O"] = rng.choice([128, 256, 512])   # the second convolution reads it as its channel count
        elif op == "lowered":
            # channel counts the implicit convolution does not take
            c.update(N=rng.randint(1, 32), H=rng.choice([14, 28, 33, 56]), C=rng.choice([16, 32, 64, 96, 192]),
                     O=_log(rng, 64, 512, 16), k=3, stride=rng.choice([1, 2]), x="relu", M=1)
        elif op == "asym":
            c.update(T=_log(rng, 1, 2048), O=width(128, 3072), I=width(128, 3072), x=rng.choice(["relu", "normal"]))
        else:
            c.update(O=width(), I=width(), pair=rng.random() < 0.3, int8_copy=rng.random() < 0.3)
        w = work(c)
        if w["flops"] <= 2.9e12 and w["bytes"] <= 1.5e9:
            return c


# ---- shapes -----------------------------------------------------------------------------------------------------------
def _keep(c: dict, O: int) -> int:
    return B.pipe_keep_groups_from_gamma(O // c["g"], c["gamma"])


def _desc(c: dict, O: int, I: int, M: int | None = None):
    return B.make_desc(O, I, c["bits"], c["K"], c["g"], _keep(c, O), c["M"] if M is None else M,
                       int8_copy=bool(c.get("int8_copy", False)))


def _rows(c: dict, O: int) -> int:
    return O + (c["K"] - 1) * _keep(c, O) * c["g"]


def _out_size(H: int, k: int, stride: int) -> int:
    return (H + 2 * (k // 2) - k) // stride + 1


def _storage_bits(c: dict) -> int:
    return {3: 4, 6: 8}.get(c["bits"], c["bits"])


def _code_bytes(c: dict, O: int, I: int) -> float:
    return _rows(c, O) * I * _storage_bits(c) / 8


def work(case: dict) -> dict:
    """Weights, inputs and outputs once each; multiply-adds of the kept rows only (an expansion: divide, round and
    update each kept element)."""
    c, op = case, case["op"]
    if op == "expand":
        total_b = total_f = 0.0
        for O, I in _expand_shapes(c):
            copies = 2 + (8 / _storage_bits(c) if c["int8_copy"] else 0)   # canonical and streaming layout (and int8)
            total_b += 4 * O * I + copies * _code_bytes(c, O, I) + 4 * _rows(c, O)
            total_f += 4 * _rows(c, O) * I
        return {"bytes": total_b, "flops": total_f}
    if op == "mlp":
        T, d, H, M = c["T"], c["I"], c["H"], c["M"]
        b = T * d * 5 + _code_bytes(c, H, d) + M * T * H * 2 + _code_bytes(c, d, H) + 4 * T * d
        return {"bytes": b, "flops": 2 * T * (d * _rows(c, H) + H * _rows(c, d))}
    if op in ("linear", "asym"):
        T, O, I, M = c["T"], c["O"], c["I"], c["M"]
        return {"bytes": M * T * I * 5 + _code_bytes(c, O, I) + 4 * M * T * O, "flops": 2 * T * I * _rows(c, O)}
    N, H, C, O, k, s = c["N"], c["H"], c["C"], c["O"], c["k"], c["stride"]
    Ho = _out_size(H, k, s)
    T1, I1 = N * Ho * Ho, k * k * C
    b, f = N * H * H * C * 5 + _code_bytes(c, O, I1), 2 * T1 * I1 * _rows(c, O)
    if op == "conv_stage":
        b += c["M"] * T1 * O * 2 + _code_bytes(c, O, k * k * O) + 4 * T1 * O
        f += 2 * T1 * k * k * O * _rows(c, O)
    else:
        b += 4 * T1 * O
    return {"bytes": b, "flops": f}


def _expand_shapes(c: dict) -> list[tuple[int, int]]:
    return [(c["O"], c["I"]), (c["I"], c["O"])] if c["pair"] else [(c["O"], c["I"])]


def tolerance(case: dict):
    # Codes, scales and kept lists of an expansion are defined bit for bit.
    if case["op"] == "expand":
        return "exact"
    # Integer sums are exact; what may differ is the order and fusing of at most eight binary32 additions per output.
    # Against the same sums in binary64: rel 4e-8 .. 7e-8, max 1.7e-7 .. 3.5e-7.
    if case["op"] not in ("mlp", "conv_stage"):
        return {"rel": 3e-7, "max": 1.5e-6}
    # Two layers: an inner code whose binary32 value lies on a rounding boundary may come out one step off.  Against a
    # binary64 evaluation of the first layer: 0 .. 1.8e-6 of the codes differ, the second layer's outputs then by rel
    # 4e-5 .. 1.6e-4, max 7e-3 .. 9e-3 (rel is about 0.13 sqrt(share)); two codes of a small layer are always allowed.
    if case["op"] == "mlp":
        n = case["T"] * case["H"]
    else:
        n = case["N"] * _out_size(case["H"], case["k"], case["stride"]) ** 2 * case["O"]
    share = max(8e-6, 2.0 / n)
    return {"rel": 0.25 * math.sqrt(share), "max": 0.04, "differ": share}


# ---- inputs -----------------------------------------------------------------------------------------------------------
def _weights(gen, c: dict, O: int, I: int) -> torch.Tensor:
    W = torch.empty((O, I), device="cuda").normal_(generator=gen)
    if c["w"] == "normal_rowmult":
        mult = torch.exp(torch.empty((O, 1), device="cuda").uniform_(math.log(0.25), math.log(4.0), generator=gen))
        return W.mul_(0.02).mul_(mult)
    if c["w"] == "student_t":   # four degrees of freedom: N / sqrt(chi2_4 / 4), chi2_4 = -2 ln(u v)
        u = torch.empty((2, O, I), device="cuda").uniform_(1e-7, 1.0, generator=gen)
        return W.mul_(0.02).div_((u[0] * u[1]).log_().mul_(-0.5).sqrt_().clamp_(min=1e-3))
    W.mul_(0.02)
    n = max(1, O * I // 1000)   # 0.1 % outliers at ten sigma
    pos = torch.randint(0, O * I, (n,), device="cuda", generator=gen)
    W.view(-1)[pos] = torch.randint(0, 2, (n,), device="cuda", generator=gen).float().mul_(0.4).sub_(0.2)
    return W


def _acts(gen, c: dict, T: int, I: int) -> torch.Tensor:
    x = torch.empty((T, I), device="cuda").normal_(generator=gen)
    if c["x"] == "relu":
        x.clamp_(min=0.0)
    elif c["x"] == "chan_outliers":
        x[:, torch.randperm(I, device="cuda", generator=gen)[:max(1, I // 200)]] *= 20.0
    return x


def _quant_buffers(T: int, I: int):
    return (torch.empty((T, I), dtype=torch.int8, device="cuda"), torch.zeros(1, device="cuda"), B.alloc_bytes(256))


def _bias(gen, O: int) -> torch.Tensor:
    return torch.empty(O, device="cuda").normal_(generator=gen).mul_(0.1)


def _geom(N: int, H: int, C: int, k: int, stride: int):
    g = B.ConvGeom()
    g.batch, g.height, g.width, g.channels = N, H, H, C
    g.kernel_h = g.kernel_w = k
    g.pad_h = g.pad_w = k // 2
    g.stride_h = g.stride_w = stride
    return g


def _step(y: torch.Tensor) -> torch.Tensor:
    """A static step for int8 outputs, calibrated on sample outputs."""
    return (y.abs().amax() / 127.0).reshape(1).float()


def prepare(case: dict, seed: int):
    c, op = case, case["op"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = {"case": c}
    if op == "expand":
        s["layers"] = []
        for O, I in _expand_shapes(c):
            desc = _desc(c, O, I)
            lay = B.pipe_layout(desc)
            blob = B.alloc_bytes(lay.blob_bytes)
            s["layers"].append((desc, _weights(gen, c, O, I), B.ExpandedLayer(desc, lay, blob), B.alloc_bytes(lay.expand_ws_bytes)))
        return s
    if op in ("linear", "asym"):
        T, O, I, M = c["T"], c["O"], c["I"], c["M"]
        s["layer"] = B.expand(_desc(c, O, I), _weights(gen, c, O, I))
        s["x"] = [_acts(gen, c, T, I) for _ in range(M)]
        s["q"] = [_quant_buffers(T, I) for _ in range(M)]
        s["zp"] = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(M)]
        s["y"] = [torch.empty((T, O), device="cuda") for _ in range(M)]
        s["bias"] = _bias(gen, O)
        return s
    if op == "mlp":
        T, d, H, M = c["T"], c["I"], c["H"], c["M"]
        s["up"], s["down"] = (B.expand(_desc(c, o, i), _weights(gen, c, o, i)) for o, i in ((H, d), (d, H)))
        s["bias"] = (_bias(gen, H), _bias(gen, d))
        # calibration of the inner step on 64 other tokens
        xs = _acts(gen, c, 64, d)
        xq, sx, ws = _quant_buffers(64, d)
        B.pipe_quantize_act(xs, xq, sx, ws)
        ys = [torch.empty((64, H), device="cuda") for _ in range(M)]
        B.pipe_ensemble_forward(s["up"].desc, s["up"].blob, [xq] * M, [sx] * M, ys, s["bias"][0])
        s["step"] = [_step(y) for y in ys]
        s["x"] = _acts(gen, c, T, d)
        s["q"] = _quant_buffers(T, d)
        s["h"] = [torch.empty((T, H), dtype=torch.int8, device="cuda") for _ in range(M)]
        s["y"] = torch.empty((T, d), device="cuda")
        return s
    N, H, C, O, k, stride = c["N"], c["H"], c["C"], c["O"], c["k"], c["stride"]
    Ho = _out_size(H, k, stride)
    T1, I1 = N * Ho * Ho, k * k * C
    s["layer"] = B.expand(_desc(c, O, I1), _weights(gen, c, O, I1))
    s["bias"] = _bias(gen, O)
    s["geom"] = _geom(N, H, C, k, stride)
    s["x"] = _acts(gen, c, N * H * H, C)
    s["q"] = _quant_buffers(N * H * H, C)
    s["y"] = torch.empty((T1, O), device="cuda")
    if op == "lowered":
        s["rows"] = torch.empty((T1, I1), dtype=torch.int8, device="cuda")
    if op == "conv_stage":
        M = c["M"]
        s["layer2"] = B.expand(_desc(c, O, k * k * O), _weights(gen, c, O, k * k * O))
        s["geom2"] = _geom(N, Ho, O, k, 1)
        xq, sx, ws = _quant_buffers(H * H, C)
        one = _geom(1, H, C, k, stride)
        B.pipe_quantize_act(_acts(gen, c, H * H, C), xq, sx, ws)
        ys = [torch.empty((Ho * Ho, O), device="cuda") for _ in range(M)]
        B.pipe_ensemble_conv2d(s["layer"].desc, one, s["layer"].blob, [xq.view(1, H, H, C)] * M, [sx] * M, ys, s["bias"])
        s["step"] = [_step(y) for y in ys]
        s["h"] = [torch.empty((T1, O), dtype=torch.int8, device="cuda") for _ in range(M)]
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------------
def run(s):
    c = s["case"]
    op = c["op"]
    if op == "expand":
        for desc, W, layer, ws in s["layers"]:
            B.pipe_expand_weights(desc, W, layer.blob, ws)
        return [[(layer.codes(k), layer.scales(k), layer.kept(k)) for k in range(c["K"])] for _, _, layer, _ in s["layers"]]
    if op == "linear":
        for x, (xq, sx, ws) in zip(s["x"], s["q"]):
            B.pipe_quantize_act(x, xq, sx, ws)
        layer = s["layer"]
        if c["M"] == 1:
            B.pipe_expanded_linear(layer.desc, layer.blob, s["q"][0][0], s["q"][0][1], s["y"][0], s["bias"])
        else:
            B.pipe_ensemble_forward(layer.desc, layer.blob, [q[0] for q in s["q"]], [q[1] for q in s["q"]], s["y"], s["bias"])
        return {"y": s["y"], "xq": [q[0] for q in s["q"]], "sx": [q[1] for q in s["q"]]}
    if op == "asym":
        for x, (xq, sx, ws), zp in zip(s["x"], s["q"], s["zp"]):
            B.pipe_quantize_act_ex(x, xq, sx, zp, ws, act_bits=8, asymmetric=True)
        layer = s["layer"]
        B.pipe_ensemble_forward_zp(layer.desc, layer.blob, [q[0] for q in s["q"]], [q[1] for q in s["q"]], s["zp"], s["y"],
                                   s["bias"])
        return {"y": s["y"], "xq": [q[0] for q in s["q"]], "sx": [q[1] for q in s["q"]], "zp": s["zp"]}
    if op == "mlp":
        M = c["M"]
        xq, sx, ws = s["q"]
        up, down = s["up"], s["down"]
        B.pipe_quantize_act(s["x"], xq, sx, ws)
        B.pipe_ensemble_forward_q8(up.desc, up.blob, [xq] * M, [sx] * M, s["step"], s["h"], s["bias"][0], ACTS[c["act"]])
        B.pipe_ensemble_forward(down.desc, down.blob, s["h"], s["step"], [s["y"]], s["bias"][1], sum_branches=True)
        return {"y": s["y"], "h": s["h"], "xq": xq, "sx": sx}
    N, H, C = c["N"], c["H"], c["C"]
    xq, sx, ws = s["q"]
    layer = s["layer"]
    B.pipe_quantize_act(s["x"], xq, sx, ws)
    xin = xq.view(N, H, H, C)
    if op == "conv":
        B.pipe_expanded_conv2d(layer.desc, s["geom"], layer.blob, xin, sx, s["y"], s["bias"])
        return {"y": s["y"], "xq": xq, "sx": sx}
    if op == "lowered":
        B.pipe_lower_conv_input(s["geom"], xin, s["rows"])
        B.pipe_expanded_linear(layer.desc, layer.blob, s["rows"], sx, s["y"], s["bias"])
        return {"y": s["y"], "xq": xq, "sx": sx}
    M, layer2, Ho = c["M"], s["layer2"], s["geom2"].height
    B.pipe_ensemble_conv2d_q8(layer.desc, s["geom"], layer.blob, [xin] * M, [sx] * M, s["step"], s["h"], s["bias"], B.ACT_RELU)
    B.pipe_ensemble_conv2d(layer2.desc, s["geom2"], layer2.blob, [h.view(N, Ho, Ho, -1) for h in s["h"]], s["step"], [s["y"]],
                           s["bias"], sum_branches=True)
    return {"y": s["y"], "h": s["h"], "xq": xq, "sx": sx}
