"""What this library is used for, as measurable cases.

Three kinds of program use it: one that packs a model's weights, one that decodes a few tokens at a time, and one that
runs many tokens through the layers (a prompt, a chunk of one, a large batch).  The shapes are those of bench.py: linear
layers of LLaMA-7B (hidden 4096, MLP 11008) and OPT-6.7B (hidden 4096, MLP 16384); token counts reach from one to 8192,
round and ragged.  Weights are heavy-tailed, activations carry a few outlier channels, as in sdq_synth.py.

A decode or prefill program holds its packed weights; most also keep the quantized-activation buffer and the outputs.
The smallest case and the one of a hundred tokens leave both to the library, as the shortest use in README.md does.
"""
from __future__ import annotations

import torch

import paper_2406_13868_b200 as sdq

# pattern and formats, by the names used below: (out_n, in_gran, in_block, scale_rule, out_fmt)
FORMATS = {
    "1of8": (1, sdq.GRAN_PAIR, 64, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),        # 1:8 FP8 outliers + pair-wise 4:8 MXFP4 (the benchmark's)
    "none": (0, sdq.GRAN_PAIR, 64, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),        # no outlier part
    "2of8": (2, sdq.GRAN_PAIR, 64, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),        # 2:8 outliers
    "block32": (1, sdq.GRAN_PAIR, 32, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),     # one scale per 32 K
    "e4m3": (1, sdq.GRAN_PAIR, 32, sdq.SCALE_UE4M3, sdq.OUT_E4M3),            # E4M3 scale codes, two-level
    "int8": (1, sdq.GRAN_PAIR, 64, sdq.SCALE_OCP_FLOOR, sdq.OUT_INT8),        # int8 outliers (grouped few-token calls)
    "elem": (1, sdq.GRAN_ELEM, 32, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),        # element-wise 2:4
    "7of8": (1, sdq.gran_keep(7), 32, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),     # 7:8 = 1:8 + 6:8, the paper's headline pattern
    "dense": (1, sdq.GRAN_DENSE, 32, sdq.SCALE_OCP_FLOOR, sdq.OUT_E4M3),      # 8:8 = 1:8 + 7:8
}
MANY_TOKEN_FORMATS = ("1of8", "none", "2of8", "block32", "e4m3", "elem", "7of8", "dense")

HIDDEN, MLP, OPT_MLP = 4096, 11008, 16384


def listed():
    return [
        # decoding one sequence: the attention output projection, a single call -- what one layer costs at the least
        {"name": "decode_o_1", "kind": "linear", "format": "1of8", "M": 1, "N": HIDDEN, "K": HIDDEN, "mats": 1},
        # decoding five sequences: gate and up read the same activations, the quantizer inside the call, the paper's int8 outliers
        {"name": "decode_gate_up_int8_5", "kind": "group_x", "format": "int8", "M": 5, "N": MLP, "K": HIDDEN, "mats": 2},
        # bench.py's decode: 32 projections of one token in one call, from the compact form of the weights
        {"name": "decode_stack32_1", "kind": "group", "format": "1of8", "M": 1, "N": HIDDEN, "K": HIDDEN, "mats": 32},
        # decoding sixteen sequences: all linear layers of one decoder layer
        {"name": "decode_layer_16", "kind": "layer", "format": "1of8", "M": 16, "K": HIDDEN, "ff": MLP},
        # a batch between decode and prefill, ragged: the gate projection
        {"name": "batch_gate_100", "kind": "linear", "format": "1of8", "M": 100, "N": MLP, "K": HIDDEN, "mats": 1},
        # a prefill chunk, ragged: q, k, v
        {"name": "chunk_qkv_500", "kind": "linear", "format": "1of8", "M": 500, "N": HIDDEN, "K": HIDDEN, "mats": 3},
        # bench.py's step: the MLP of one layer at prefill
        {"name": "prefill_mlp_2048", "kind": "mlp", "format": "1of8", "M": 2048, "K": HIDDEN, "ff": MLP, "gated": True},
        # the largest: all linear layers of one decoder layer, 8192 tokens
        {"name": "prefill_layer_8192", "kind": "layer", "format": "1of8", "M": 8192, "K": HIDDEN, "ff": MLP},
        # OPT's two-layer MLP at prefill with E4M3 scales per 32 K, the best scale format of the paper's study
        {"name": "prefill_opt_e4m3_4096", "kind": "mlp", "format": "e4m3", "M": 4096, "K": HIDDEN, "ff": OPT_MLP, "gated": False},
        # the paper's headline pattern (inliers stored dense) at a ragged prompt length: the down projection
        {"name": "prefill_down_7of8_1500", "kind": "linear", "format": "7of8", "M": 1500, "N": HIDDEN, "K": MLP, "mats": 1},
        # packing for a decode deployment: decompose a gate projection, keep the compact form too
        {"name": "pack_gate", "kind": "pack", "format": "1of8", "N": MLP, "K": HIDDEN, "calib": 0},
        # packing with the weight-activation product metric: channel norms of a calibration batch, then decompose
        {"name": "pack_down_7of8_metric", "kind": "pack", "format": "7of8", "N": HIDDEN, "K": MLP, "calib": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _dim(rng, step, lo, hi):
    return max(lo, min(hi, step * round(_log_int(rng, lo, hi) / step)))


def draw(rng):
    kind = rng.choice(("linear", "linear", "group", "group_x", "layer", "mlp", "pack"))
    K = _dim(rng, 256, 1024, 16384)
    if kind == "linear":
        # one to three projections of the same activations, one call after the other, any number of tokens
        return {"kind": kind, "format": rng.choice(MANY_TOKEN_FORMATS), "M": _log_int(rng, 1, 8192), "N": _dim(rng, 128, 1024, 16384),
                "K": K, "mats": rng.randint(1, 3)}
    if kind == "group":
        mats = _log_int(rng, 2, 32)
        return {"kind": kind, "format": rng.choice(("1of8", "int8")), "M": _log_int(rng, 1, 32), "N": _dim(rng, 128, max(1024, 128 * -(-80 // mats)), 11008),
                "K": min(K, 11008), "mats": mats}
    if kind == "group_x":
        mats = rng.randint(2, 4)
        return {"kind": kind, "format": rng.choice(("1of8", "int8")), "M": _log_int(rng, 1, 16), "N": _dim(rng, 128, 5120, 16384),
                "K": _dim(rng, 256, 1024, 4096), "mats": mats}
    if kind == "pack":
        return {"kind": kind, "format": rng.choice(("1of8", "2of8", "block32", "e4m3", "int8", "elem", "7of8", "dense")), "N": _dim(rng, 128, 1024, 16384),
                "K": K, "calib": rng.choice((0, _log_int(rng, 128, 4096)))}
    # a decoder layer or its MLP: hidden size and MLP width of models of 1 to 13 billion weights, any number of tokens
    K = _dim(rng, 256, 2048, 4096)
    ff = _dim(rng, 256, 2 * K, 11008)
    M = _log_int(rng, 1, 8000)
    if kind == "mlp":
        return {"kind": kind, "format": rng.choice(MANY_TOKEN_FORMATS), "M": M, "K": K, "ff": ff, "gated": rng.random() < 0.5}
    return {"kind": kind, "format": "1of8", "M": M, "K": K, "ff": ff}


def _config(case):
    out_n, gran, block, rule, fmt = FORMATS[case["format"]]
    return sdq.Config(out_n, gran, block, rule, sdq.ORDER_LARGE, fmt)


def _weight(N, K, g):
    """Student-t (4 degrees of freedom) weights of scale 0.02, in bf16"""
    w = torch.empty((N, K), dtype=torch.bfloat16, device="cuda")
    rows = max(1, (1 << 24) // K)
    for r in range(0, N, rows):
        n = min(rows, N - r)
        z = torch.randn((n, K), generator=g, device="cuda")
        u = torch.rand((2, n, K), generator=g, device="cuda").clamp_min_(1e-30)
        w[r:r + n] = (z * torch.sqrt(-2.0 / torch.log(u[0] * u[1])) * 0.02).to(torch.bfloat16)
    return w


def _act(M, K, g):
    """N(0, 1) activations in bf16, one channel of 128 thirty times as large"""
    x = torch.randn((M, K), generator=g, device="cuda")
    x[:, torch.randperm(K, generator=g, device="cuda")[: max(1, K // 128)]] *= 30.0
    return x.to(torch.bfloat16)


def _shapes(case):
    """(N, K) of the weight matrices of one pass"""
    if case["kind"] == "layer":
        K, ff = case["K"], case["ff"]
        return [(K, K)] * 4 + [(ff, K)] * 2 + [(K, ff)]
    if case["kind"] == "mlp":
        K, ff = case["K"], case["ff"]
        return [(ff, K)] * (2 if case["gated"] else 1) + [(K, ff)]
    return [(case["N"], case["K"])] * case.get("mats", 1)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind, cfg = case["kind"], _config(case)
    s = {"kind": kind, "cfg": cfg}
    if kind == "pack":
        s["W"] = _weight(case["N"], case["K"], g)
        s["calib"] = _act(case["calib"], case["K"], g) if case["calib"] else None
        return s
    M = case["M"]
    s["P"] = [sdq.sdq_decompose(_weight(N, K, g), cfg) for N, K in _shapes(case)]
    if kind == "group":
        s["P"] = [sdq.packed_compact(p) for p in s["P"]]
    s["X"] = _act(M, case["K"], g)
    if kind in ("layer", "mlp"):
        s["H"] = _act(M, case["ff"], g)
        s["hbuf"] = torch.empty(sdq.act_size(M, case["ff"], cfg), dtype=torch.uint8, device="cuda")
    if kind == "layer":
        s["X2"], s["X3"] = _act(M, case["K"], g), _act(M, case["K"], g)
        s["grouped"] = M <= 32
    if kind != "linear":
        s["xbuf"] = torch.empty(sdq.act_size(M, case["K"], cfg), dtype=torch.uint8, device="cuda")
        s["Y"] = [torch.empty((M, p.N), dtype=torch.bfloat16, device="cuda") for p in s["P"]]
    return s


def run(s):
    kind, cfg = s["kind"], s["cfg"]
    if kind == "pack":
        if s["calib"] is not None:
            return sdq.sdq_decompose(s["W"], cfg, col_weight=sdq.channel_norm(s["calib"])).buf
        p = sdq.sdq_decompose(s["W"], cfg)
        return [p.buf, sdq.packed_compact(p).buf]
    P = s["P"]
    if kind == "linear":
        xq = sdq.sdq_quantize_act(s["X"], cfg)
        return [sdq.sdq_linear(xq, p) for p in P]
    Y = s["Y"]
    if kind == "group_x":
        return sdq.sdq_linear_group_x(s["X"], P, Y)
    xq = sdq.sdq_quantize_act(s["X"], cfg, s["xbuf"])
    if kind == "group":
        return sdq.sdq_linear_group([xq] * len(P), P, Y)
    if kind == "mlp":
        for p, y in zip(P[:-1], Y):
            sdq.sdq_linear(xq, p, y)
        sdq.sdq_linear(sdq.sdq_quantize_act(s["H"], cfg, s["hbuf"]), P[-1], Y[-1])
        return Y
    # a decoder layer: q, k, v | o | gate, up | down, each group behind its own activations
    if s["grouped"]:
        sdq.sdq_linear_group([xq] * 3, P[0:3], Y[0:3])
    else:
        for i in (0, 1, 2):
            sdq.sdq_linear(xq, P[i], Y[i])
    sdq.sdq_linear(sdq.sdq_quantize_act(s["X2"], cfg, s["xbuf"]), P[3], Y[3])
    xq = sdq.sdq_quantize_act(s["X3"], cfg, s["xbuf"])
    if s["grouped"]:
        sdq.sdq_linear_group([xq] * 2, P[4:6], Y[4:6])
    else:
        for i in (4, 5):
            sdq.sdq_linear(xq, P[i], Y[i])
    sdq.sdq_linear(sdq.sdq_quantize_act(s["H"], cfg, s["hbuf"]), P[6], Y[6])
    return Y


def work(case):
    cfg, shapes = _config(case), _shapes(case)
    if case["kind"] == "pack":
        # the weights (and calibration activations) once in, the packed buffer once out; its compact form once more where it is kept
        N, K = case["N"], case["K"]
        full, algorithmic = sdq.packed_size(N, K, cfg)
        return {"bytes": 2 * N * K + full + (2 * case["calib"] * K if case["calib"] else algorithmic), "flops": 0}
    M = case["M"]
    inputs = {"layer": 3 * case["K"] + case.get("ff", 0), "mlp": case["K"] + case.get("ff", 0)}.get(case["kind"], case["K"])
    weights = sum(sdq.packed_size(N, K, cfg)[1] for N, K in shapes)
    return {"bytes": 2 * M * inputs + weights + sum(2 * M * N for N, _ in shapes), "flops": sum(2 * M * N * K for N, K in shapes)}


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    # bf16 outputs of fp32 sums of exact products: another order of the sums moves a value in a million to the neighbouring
    # bf16 number (2^-7 of the value at most; against the exact sums: rel 6e-6 over 2 million outputs), which is more of
    # the whole where there are few outputs
    return {"rel": 1e-4, "max": 8e-3}
