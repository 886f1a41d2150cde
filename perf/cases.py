"""The subgraphs whose speed counts, as a user's program runs them: a handle made once, its weights on the GPU, and
then one `Subgraph.run(inputs, weights)` per batch, on the current stream, the result in a new tensor.

A case is a chain family with its sizes and the execution mode. Every family of the library occurs: inverted-residual
blocks and their two-operator pairs, residual blocks of 3x3 convolutions, attention, feed-forward chains, the
patch-unfolded projection pair and the stand-alone depthwise stage in 32-bit floats. The listed cases are the
benchmark's configurations (`paper_2212_01005_b200/workloads.py`) and, beside them, the sizes such chains have where
nothing was tuned: short and ragged sequences, odd images, wide blocks, row counts that are no multiple of a tile.
`draw` spreads over the same ranges. The library runs a subgraph in one direction; it has no backward pass.
"""
from __future__ import annotations

import math

import torch

from paper_2212_01005_b200 import binding as B
from paper_2212_01005_b200 import workloads as WL

# Bounds of a drawn case, per pass: the largest listed case is at 116 GFLOP.
MOST_FLOPS = 1.0e11
MOST_BYTES = 2.0e8


def listed():
    return [
        # Latency of one request: a 14x14 inverted-residual block of a single image.
        {"name": "block_14_one_image", "family": "block", "mode": "fused", "n": 1, "h": 14, "w": 14, "cin": 32, "cexp": 192,
         "cout": 32, "stride": 1, "residual": True},
        # Batched image classification, early block: large maps, few channels, residual.
        {"name": "block_56_batch_32", "family": "block", "mode": "fused", "n": 32, "h": 56, "w": 56, "cin": 24, "cexp": 144,
         "cout": 24, "stride": 1, "residual": True},
        # The block that halves the map between two stages.
        {"name": "block_28_stride_2", "family": "block", "mode": "fused", "n": 32, "h": 28, "w": 28, "cin": 32, "cexp": 192,
         "cout": 64, "stride": 2, "residual": False},
        # A late, wide block (96 channels, expanded six times) on an odd map and batch; the planner chooses how to run it.
        {"name": "block_wide_odd", "family": "block", "mode": "auto", "n": 25, "h": 15, "w": 15, "cin": 96, "cexp": 576,
         "cout": 96, "stride": 1, "residual": True},
        # A residual block of two 3x3 convolutions in the first stage of a batched image network.
        {"name": "residual_56_batch_32", "family": "residual", "mode": "fused", "n": 32, "h": 56, "w": 56, "c": 64},
        # Encoder attention over full-length sequences.
        {"name": "attention_384", "family": "attention", "mode": "fused", "n": 32, "s": 384, "heads": 12},
        # Encoder attention of a small batch of shorter sequences whose length is no multiple of a tile.
        {"name": "attention_200_small", "family": "attention", "mode": "auto", "n": 3, "s": 200, "heads": 12},
        # Feed-forward chain of a small token batch.
        {"name": "feed_forward_512", "family": "feed_forward", "mode": "auto", "rows": 512, "d": 768, "hidden": 3072},
        # Feed-forward chain of a medium, ragged token batch; the planner chooses how to run it.
        {"name": "feed_forward_ragged", "family": "feed_forward", "mode": "auto", "rows": 3001, "d": 768, "hidden": 3072},
        # Feed-forward chain of 32 sequences of 384 tokens in one fused pass: the largest configuration.
        {"name": "feed_forward_12288", "family": "feed_forward", "mode": "fused", "rows": 12288, "d": 768, "hidden": 3072},
        # Two depthwise stages in a row at the memory-bound end of the operator pairs.
        {"name": "pair_dw_dw_56", "family": "dw_dw", "mode": "fused", "n": 32, "h": 56, "w": 56, "c": 144},
        # Projections around the patch transpose of a mobile vision transformer.
        {"name": "unfold_96", "family": "unfold", "mode": "fused", "n": 32, "p": 4, "patches": 256, "d": 96, "d_out": 192},
    ]


def _log(rng, low, high):
    """A whole number from low to high, spread over its logarithm."""
    return min(high, max(low, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    """Each family about as often as it is listed, the pairs and the 32-bit stage once more; sizes over the whole range."""
    while True:
        case = _draw(rng)
        cost = work(case)
        if cost["flops"] <= MOST_FLOPS and cost["bytes"] <= MOST_BYTES:
            return case


def _draw(rng):
    family = rng.choice(["block"] * 4 + ["residual"] * 2 + ["attention"] * 3 + ["feed_forward"] * 4 +
                        ["pw_dw", "dw_pw", "dw_dw", "pw_pw", "unfold", "depthwise32"])
    mode = "auto"
    if family == "block":
        # stages of 7 to 112 pixels; the wider the block, the smaller its map
        cin = rng.choice([16, 24, 32, 40, 64, 96, 160])
        h = _log(rng, 7, {16: 112, 24: 64, 32: 48, 40: 32, 64: 28, 96: 20, 160: 14}[cin])
        stride = rng.choice([1, 1, 2])
        residual = stride == 1 and rng.random() < 0.6
        cout = cin if residual else rng.choice([c for c in (16, 24, 32, 64, 96, 160) if cin // 2 <= c <= 3 * cin])
        return {"family": family, "mode": mode, "n": _log(rng, 1, 64), "h": h, "w": h, "cin": cin, "cexp": 6 * cin, "cout": cout,
                "stride": stride, "residual": residual}
    if family == "residual":
        h = _log(rng, 9, 80)
        return {"family": family, "mode": mode, "n": _log(rng, 1, 48), "h": h, "w": max(9, h + rng.randint(-3, 3)), "c": rng.choice([16, 32, 64, 64])}
    if family == "attention":
        s = 8 * rng.randint(4, 48)
        return {"family": family, "mode": mode, "n": _log(rng, 1, max(1, 12288 // s)), "s": s, "heads": rng.choice([2, 4, 8, 12, 16])}
    if family == "feed_forward":
        d = rng.choice([256, 384, 512, 768, 768, 1024])
        return {"family": family, "mode": rng.choice(["auto", "auto", "fused"]), "rows": _log(rng, 1, 12288), "d": d, "hidden": 4 * d}
    if family == "unfold":
        d = rng.choice([32, 48, 64, 96, 120])
        return {"family": family, "mode": mode, "n": _log(rng, 1, 64), "p": rng.choice([4, 9, 16]), "patches": rng.randint(4, 18) ** 2, "d": d, "d_out": 2 * d}
    h = _log(rng, 7, 64)
    case = {"family": family, "mode": mode, "n": _log(rng, 1, 48), "h": h, "w": h, "c": 16 * rng.randint(3, 12)}
    if family != "depthwise32":
        case["narrow"] = rng.choice([16, 24, 32, 40])     # the other width of a pair (unused between two depthwise stages)
    if family in ("pw_dw", "dw_pw", "depthwise32"):
        case["stride"] = rng.choice([1, 1, 2])
    return case


def _workload(case):
    c, family = case, case["family"]
    name = family
    if family == "block":
        ops = WL._mbv2_ops(c["cexp"], c["cout"], c["stride"], c["residual"])
        return WL.Workload(name, [0], [(c["n"], c["h"], c["w"], c["cin"])], ops, samples=c["n"], input_dist=["uniform"])
    if family == "residual":
        return WL.Workload(name, [0], [(c["n"], c["h"], c["w"], c["c"])], WL._resnet_ops(c["c"]), samples=c["n"], input_dist=["relu_normal"])
    if family == "attention":
        return WL.attention(name, [0], c["n"], c["s"], c["heads"], 64)
    if family == "feed_forward":
        return WL.ffn(name, [0], c["rows"], c["d"], c["hidden"], samples=1)
    if family == "unfold":
        return WL.unfold_chain(name, [0], c["n"], c["p"], c["patches"], c["d"], c["d_out"])
    if family == "pw_dw":
        return WL.pw_dw(name, [0], c["n"], c["h"], c["narrow"], c["c"], c["stride"])
    if family == "dw_pw":
        return WL.dw_pw(name, [0], c["n"], c["h"], c["c"], c["narrow"], c["stride"])
    if family == "dw_dw":
        return WL.dw_dw(name, [0], c["n"], c["h"], c["c"])
    if family == "pw_pw":
        return WL.pw_pw(name, [0], c["n"], c["h"], c["c"], c["narrow"], c["c"])
    if family == "depthwise32":
        ops = [("conv2d", dict(O=c["c"], R=3, S=3, stride=c["stride"], pad=1, groups=c["c"])), ("bias_add", {}), ("relu6", {})]
        return WL.Workload(name, [0], [(c["n"], c["h"], c["w"], c["c"])], ops, samples=c["n"], input_dist=["uniform"])
    raise ValueError(family)


def prepare(case, seed):
    """Inputs and weights with the distributions of `workloads.generate`, drawn on the GPU, and the handle with its workspace."""
    wl = _workload(case)
    fp32 = case["family"] == "depthwise32"
    dtype = torch.float32 if fp32 else torch.bfloat16
    device = torch.device("cuda")
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed))
    inputs, weights = [], []
    for shape, dist in zip(wl.input_shapes, wl.input_dist):
        if dist == "uniform":
            t = torch.rand(shape, generator=gen, device=device) * 2.0 - 1.0
        else:
            t = torch.randn(shape, generator=gen, device=device)
            if dist == "relu_normal":
                t = t.clamp_min_(0.0)
        inputs.append(t.to(dtype))
    gain = 2.0 if wl.ops[0][0] == "conv2d" else 1.0
    for shape, kind, fan in zip(wl.weight_shapes, wl.weight_kinds, wl.weight_fan_in):
        if kind == "bias":
            weights.append(torch.rand(shape, generator=gen, device=device) * 0.2 - 0.1)
        else:
            weights.append((torch.randn(shape, generator=gen, device=device) * math.sqrt(gain / fan)).to(dtype))
    handle = B.Subgraph(wl.ops, wl.input_shapes, mode=case["mode"], dtype=B.AGO_FP32 if fp32 else B.AGO_BF16)
    handle.ensure_workspace(inputs[0].device)
    return handle, inputs, weights


def run(state):
    handle, inputs, weights = state
    return handle.run(inputs, weights)


def work(case):
    wl = _workload(case)
    flops = WL.flops(wl)
    scale = 2 if case["family"] == "depthwise32" else 1     # io_bytes counts activations and weights in bf16
    return {"bytes": scale * WL.io_bytes(wl), "flops": flops["tensor"] + flops["cuda"]}


def tolerance(case):
    """Four times what the library differs by from the chain in 64-bit floats (rel 2.0e-3 to 3.0e-3 and max 0.6e-2 to 2.2e-2
    over all families in bf16: the rounding of the intermediates a tensor-core operand needs and of the output;
    rel 6e-8 and max 4e-7 for the 32-bit depthwise stage: the order of nine products)."""
    if case["family"] == "depthwise32":
        return {"rel": 5e-7, "max": 4e-6}
    return {"rel": 1.0e-2, "max": 0.08}
