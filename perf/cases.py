"""The workloads whose speed is followed: what a program that uses libmsla asks of it.

An inference program holds the weights, a descriptor and a workspace, and calls one of four entry points per feature
map: the multi-scale linear attention module (``msla_forward``, or ``msla_forward_host`` where the activations live on
the host), the attention core on its own (``msla_linattn_relu_ws``), or the whole building block
(``msla_evit_block``: the module and the FFN with a depthwise convolution).  The library is forward-only.

The ranges: token grids from 7x7 (the last stage of a 224-pixel classifier) to 512x512, one image to a batch of 64,
64 to 384 channels, heads of 16 and 32 channels, bf16 and fp16 storage (deployment) and fp32 (checking and
unquantised use), with and without a bias on the output projection (a folded normalisation).  Grids are whatever the
image size gives, so their token counts are often no multiple of anything.
"""
from __future__ import annotations

import math

import torch

from paper_2205_14756_b200 import binding

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
EPS = 1e-15
LARGEST_FLOPS = 240e9       # the 512x512 module
LARGEST_F32_TOKEN_CHANNELS = 64 * 128 * 192


def _module(name, dtype, B, C, H, W, d, bias=False):
    return {"name": name, "op": "module", "dtype": dtype, "B": B, "C": C, "H": H, "W": W, "d": d, "bias": bias}


def listed():
    return [
        # one small feature map, the narrowest module, full precision: a call is all launches and latency
        _module("module_f32_b1_16x16_c64_d16", "f32", 1, 64, 16, 16, 16),
        # stride-16 features of a 1024x2048 street scene kept in fp32 (checking a quantised deployment against it)
        _module("module_f32_b1_64x128_c192_d32", "f32", 1, 192, 64, 128, 32),
        # stride-16 features of one 512x512 image: the latency of a single call
        _module("module_bf16_b1_32x32_c256_d32", "bf16", 1, 256, 32, 32, 32),
        # stride-16 features of a 1024x2048 street scene
        _module("module_bf16_b1_64x128_c192_d32", "bf16", 1, 192, 64, 128, 32),
        # stride-16 features of a batch of 1024x1024 images
        _module("module_bf16_b16_64x64_c256_d32", "bf16", 16, 256, 64, 64, 32),
        # the high-resolution end: 262 144 tokens of one image
        _module("module_bf16_b1_512x512_c256_d32", "bf16", 1, 256, 512, 512, 32),
        # classification: stride-16 features of a batch of 224-pixel images, 196 tokens each (not a multiple of 8)
        _module("module_bf16_b64_14x14_c256_d32", "bf16", 64, 256, 14, 14, 32),
        # fp16 deployment with narrow heads and a folded normalisation: stride-16 features of 720x1280 video frames
        _module("module_f16_b8_45x80_c128_d16", "f16", 8, 128, 45, 80, 16, bias=True),
        # the attention core alone, for programs with projections of their own: 64x64 tokens, 16 heads
        {"name": "core_bf16_b8_h16_n4096_d32", "op": "core", "dtype": "bf16", "B": 8, "heads": 16, "N": 4096, "d": 32},
        # the whole building block on stride-8 features of a 1024x2048 street scene, expansion 4
        {"name": "block_bf16_b1_128x256_c256_h1024", "op": "block", "dtype": "bf16", "B": 1, "C": 256, "H": 128, "W": 256,
         "d": 32, "hidden": 1024},
        # the block in the last stages of a fp16 classifier: stride-8 features of a few 224-pixel images
        {"name": "block_f16_b4_28x28_c128_h512", "op": "block", "dtype": "f16", "B": 4, "C": 128, "H": 28, "W": 28,
         "d": 16, "hidden": 512},
        # activations in pinned host memory, a batch per call, the result back on the host
        {"name": "host_bf16_b16_64x64_c256_d32", "op": "host", "dtype": "bf16", "B": 16, "C": 256, "H": 64, "W": 64, "d": 32,
         "bias": False},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges; grid sides are any integers, batches and widths follow from what fits."""
    while True:
        op = rng.choices(["module", "core", "block", "host"], weights=[7, 2, 2, 1])[0]
        dtype = rng.choices(["bf16", "f16", "f32"], weights=[6, 3, 2])[0]
        d = rng.choice([16, 32, 32])
        B = _log_int(rng, 1, 64)
        H = _log_int(rng, 7, 512)
        W = min(512, max(7, int(round(H * math.exp(rng.uniform(-0.9, 0.9))))))
        if op == "core":
            case = {"op": op, "dtype": dtype, "B": B, "heads": rng.randint(2, 24), "N": H * W, "d": d}
            width = 3 * case["heads"] * d
        else:
            C = 32 * rng.randint(2, 12)
            case = {"op": op, "dtype": dtype, "B": B, "C": C, "H": H, "W": W, "d": d}
            width = C
            if op == "block":
                case["hidden"] = 4 * C
            else:
                case["bias"] = rng.random() < 0.5
        need = work(case)
        tokens = B * H * W
        if need["flops"] > LARGEST_FLOPS or need["bytes"] > 540e6:
            continue
        if dtype == "f32" and tokens * width > LARGEST_F32_TOKEN_CHANNELS:
            continue
        if op == "host" and need["bytes"] > 80e6:
            continue
        return case


def prepare(case, seed):
    """Seeded inputs and weights on the GPU, and the descriptor and workspace a program keeps from call to call.
    Activations ~ N(0, 1), weights ~ N(0, 1 / fan_in), biases ~ N(0, 1/4)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = DTYPES[case["dtype"]]
    code = binding.dtype_code(dt)

    def normal(*shape, std=1.0):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32).mul_(std).to(dt)

    def scratch(nbytes):
        return torch.empty(nbytes, dtype=torch.uint8, device="cuda")

    B, d = case["B"], case["d"]
    if case["op"] == "core":
        heads, N = case["heads"], case["N"]
        q, k, v = (normal(B, heads, N, d) for _ in range(3))
        nbytes = binding.msla_linattn_relu_workspace_bytes(B, heads, N, d)
        return {"op": "core", "code": code, "q": q, "k": k, "v": v, "out": torch.empty_like(q), "B": B, "heads": heads, "N": N,
                "d": d, "ws": scratch(nbytes), "ws_bytes": nbytes}

    C, H, W = case["C"], case["H"], case["W"]
    heads = C // d
    x = normal(B, C, H, W)
    keep = {"w_qkv": normal(3 * C, C, std=C ** -0.5), "w_dw": normal(3 * C, 5, 5, std=0.2),
            "w_pw": normal(3 * C, d, std=d ** -0.5), "w_proj": normal(C, 2 * C, std=(2 * C) ** -0.5),
            "b_proj": normal(C, std=0.5) if case.get("bias") else None}
    weights = binding.make_weights(keep["w_qkv"], keep["w_dw"], keep["w_pw"], keep["w_proj"], keep["b_proj"])
    plain = binding.make_desc(B, C, H, W, heads, d, C, code, EPS)
    state = {"op": case["op"], "keep": keep, "weights": weights, "x": x, "out": torch.empty_like(x)}
    if case["op"] == "host":
        ws = scratch(binding.msla_forward_host_workspace_bytes(plain))
        state["x"], state["out"] = x.cpu().pin_memory(), torch.empty(B, C, H, W, dtype=dt, pin_memory=True)
    else:
        ws = scratch(binding.msla_forward_workspace_bytes(plain))
    state["ws"] = ws
    state["desc"] = binding.make_desc(B, C, H, W, heads, d, C, code, EPS, workspace=ws)
    if case["op"] == "block":
        hidden = case["hidden"]
        keep.update(w1=normal(hidden, C, std=C ** -0.5), b1=normal(hidden, std=0.5), w_ffn_dw=normal(hidden, 3, 3, std=1 / 3),
                    b_ffn_dw=normal(hidden, std=0.5), w2=normal(C, hidden, std=hidden ** -0.5), b2=normal(C, std=0.5))
        state["ffn_weights"] = binding.make_ffn_weights(keep["w1"], keep["w_ffn_dw"], keep["w2"], keep["b1"], keep["b_ffn_dw"], keep["b2"])
        plain = binding.make_ffn_desc(B, C, H, W, hidden, C, code, binding.MSLA_ACT_HARDSWISH, residual=True)
        state["ffn_ws"] = scratch(binding.msla_ffn_workspace_bytes(plain))
        state["ffn_desc"] = binding.make_ffn_desc(B, C, H, W, hidden, C, code, binding.MSLA_ACT_HARDSWISH, residual=True,
                                                  workspace=state["ffn_ws"])
        state["y"] = torch.empty_like(x)
    return state


def run(state):
    """One call, on the current stream."""
    op = state["op"]
    if op == "core":
        binding.msla_linattn_relu_ws(state["code"], state["q"], state["k"], state["v"], state["out"], state["B"], state["heads"],
                                     state["N"], state["d"], EPS, state["ws"], state["ws_bytes"])
        return state["out"]
    if op == "block":
        binding.msla_evit_block(state["desc"], state["weights"], state["ffn_desc"], state["ffn_weights"], state["x"], state["y"],
                                state["out"])
        return {"attention": state["y"], "out": state["out"]}
    if op == "host":
        binding.msla_forward_host(state["desc"], state["x"], state["weights"], state["out"])
        torch.cuda.current_stream().synchronize()  # the caller reads the result on the host
        return state["out"]
    binding.msla_forward(state["desc"], state["x"], state["weights"], state["out"])
    return state["out"]


def work(case):
    """Bytes: the call's inputs (activations and weights) read once, its outputs written once.  Flops: the five steps
    (and the FFN's three) as they are defined, two per multiply-add, the d x d contractions of Eq. 3 among them."""
    e = 4 if case["dtype"] == "f32" else 2
    B, d = case["B"], case["d"]
    if case["op"] == "core":
        rows = B * case["heads"] * case["N"]
        return {"bytes": 4 * rows * d * e, "flops": 4 * rows * d * (d + 1)}
    C = case["C"]
    tokens = B * case["H"] * case["W"]
    params = 3 * C * C + 3 * C * 25 + 3 * C * d + 2 * C * C
    per_token = 3 * C * C + 3 * C * (25 + d) + 2 * (2 * C * (d + 1)) + 2 * C * C
    outputs = 1
    if case["op"] == "block":
        hidden = case["hidden"]
        params += 2 * hidden * C + 11 * hidden + C
        per_token += 2 * hidden * C + 9 * hidden
        outputs = 2
    return {"bytes": ((1 + outputs) * tokens * C + params) * e, "flops": 2 * tokens * per_token}


def tolerance(case):
    """Relative 2-norm error; about four times what the library shows against the same path in 64 bits
    (measured: fp32 up to 5.0e-7, bf16 up to 3.7e-3, fp16 up to 3.0e-4)."""
    return {"rel": {"f32": 2.5e-6, "bf16": 1.4e-2, "f16": 1.2e-3}[case["dtype"]]}
