"""The work that a user of libunitscale has it do, as a list of measurable cases.

`listed()` names them, `draw(rng)` gives one more of the same ranges.  `prepare(case, seed)` makes what a program holds
before the call (seeded inputs on the GPU, the block or layer object, the workspace, for `graph` cases the captured
step), `run(state)` is one pass through the public entry points and returns all of its results, `work(case)` says what
a pass cannot do without, `tolerance(case)` how far another correct implementation of the same precision may be off.

Kinds of work:
  step     one training step of the FFN block: casts, forward, backward (`UnitScaledFFN.step`, or its captured graph)
  forward  evaluation of the FFN block with its weights already quantised (`UnitScaledFFN.forward`)
  encoder  one training step of an encoder layer (`UnitScaledEncoderLayer.step`)
  linear   one linear layer on its own: forward, input gradient, weight gradient (`us_linear_fwd / bwd_x / bwd_w`)
  head     an output projection with its loss: quantise, logits, softmax cross-entropy forward and backward, both
           gradients of the projection

All inputs are N(0, 1), the distribution unit scaling keeps activations, weights and gradients at.
"""
import math

import torch

from paper_2303_11257_b200 import encoder, ffn
from paper_2303_11257_b200 import lib as L

E4, E5 = torch.float8_e4m3fn, torch.float8_e5m2
OPERANDS = {"fp8": (E4, E5), "bf16": (torch.bfloat16, torch.bfloat16), "fp16": (torch.float16, torch.float16)}
OUTPUTS = {"f32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16, "e4m3": E4, "e5m2": E5}


def _step(tokens, d, f, operand="fp8", graph=True):
    return {"kind": "step", "tokens": tokens, "d": d, "f": f, "operand": operand, "graph": graph}


def _encoder(nseq, slen, nhead, attention, fused, norm):
    return {"kind": "encoder", "nseq": nseq, "slen": slen, "nhead": nhead, "attention": attention, "fused": fused, "norm": norm}


def listed():
    cases = {
        # character language model (hidden 128, FFN 512, sequence 256): the smallest step, called as a script calls it ...
        "step_char_lm": _step(256, 128, 512, graph=False),
        # ... and as a training loop replays it
        "step_char_lm_graph": _step(256, 128, 512),
        # sizes that are multiples of no tile (a sub-batch left over at the end of an epoch, a pruned width)
        "step_ragged": _step(1000, 528, 2096, graph=False),
        # the FFN block of BERT-large on 16 x 512 tokens: the repository's benchmark, FP8 and its 16-bit alternative
        "step_bert_large_fp8": _step(8192, 1024, 4096),
        "step_bert_large_bf16": _step(8192, 1024, 4096, "bf16"),
        # a wider block on twice the tokens: the largest step
        "step_wide": _step(16384, 2048, 8192),
        # evaluation of a few sentences with a trained block
        "forward_few_tokens": {"kind": "forward", "tokens": 48, "d": 1024, "f": 4096, "operand": "fp8"},
        # one BERT-large layer on 16 x 512 tokens, fused attention: 16-bit attention operands without layer norms
        # (the repository's encoder benchmark), and every matmul in FP8 with the post-norm arrangement
        "encoder_bert_large_bf16": _encoder(16, 512, 16, "bf16", True, ""),
        "encoder_bert_large_fp8_norm": _encoder(16, 512, 16, "fp8", True, "post"),
        # a layer of the character language model as the class builds it by default
        "encoder_char_lm": _encoder(8, 256, 2, "bf16", False, ""),
        # one large projection on a short batch (the skinny shape of the repository's GEMM sweep)
        "linear_skinny": {"kind": "linear", "b": 512, "m": 8192, "n": 8192, "operand": "fp8", "out": "bf16"},
        # masked-language-model head: 2048 predicted tokens, a vocabulary of 30522
        "head_vocabulary": {"kind": "head", "tokens": 2048, "d": 1024, "classes": 30522},
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log(rng, lo, hi, multiple=1):
    """An integer of [lo, hi], spread over its logarithm, rounded to a multiple."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(max(int(round(v / multiple)), -(-lo // multiple)), hi // multiple) * multiple


_MOST_FLOPS = 12.0 * 16384 * 2048 * 8192


def draw(rng):
    kind = rng.choice(["step"] * 8 + ["forward"] * 2 + ["encoder"] * 4 + ["linear"] * 4 + ["head"] * 2)
    while True:
        if kind == "step":
            d = _log(rng, 128, 2048, 16)
            c = _step(_log(rng, 16, 16384), d, min(8192, _log(rng, 2 * d, 4 * d, 16)), rng.choice(["fp8", "fp8", "fp8", "bf16", "fp16"]), rng.random() < 0.5)
        elif kind == "forward":
            d = _log(rng, 128, 2048, 16)
            c = {"kind": kind, "tokens": _log(rng, 1, 8192), "d": d, "f": _log(rng, 2 * d, 4 * d, 16), "operand": rng.choice(["fp8", "fp8", "bf16"])}
        elif kind == "encoder":
            slen = _log(rng, 16, 1024, 16)
            c = _encoder(max(1, _log(rng, 256, 8192) // slen), slen, rng.choice([2, 3, 4, 6, 8, 12, 16]), rng.choice(["bf16", "fp8", "fp16"]),
                         slen <= 512 and rng.random() < 0.75, rng.choice(["", "post"]))
        elif kind == "linear":
            c = {"kind": kind, "b": _log(rng, 16, 16384), "m": _log(rng, 128, 8192, 16), "n": _log(rng, 128, 8192, 16),
                 "operand": rng.choice(["fp8", "fp8", "bf16", "fp16"]), "out": rng.choice(["bf16", "f32", "e4m3"])}
        else:
            c = {"kind": kind, "tokens": _log(rng, 64, 4096), "d": _log(rng, 128, 1024, 16), "classes": _log(rng, 1000, 40000)}
        if work(c)["flops"] <= _MOST_FLOPS:
            return c


def _normal(seed, shapes):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    return [torch.randn(s, generator=g, device="cuda") for s in shapes]


def _padded(rows, cols, dtype):
    """rows x cols with a row pitch of a multiple of 16 elements, as the library's alignment rule wants it."""
    return torch.empty((rows, (cols + 15) // 16 * 16), dtype=dtype, device="cuda")[:, :cols]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("step", "forward"):
        T, d, f = case["tokens"], case["d"], case["f"]
        s["x"] = _normal(seed, [(T, d), (d, f), (f, d), (T, d)])
        s["block"] = ffn.UnitScaledFFN(T, d, f, operand=case["operand"])
        if kind == "forward":
            s["block"].cast_weights(s["x"][1], s["x"][2])
        elif case["graph"]:
            s["block"].step(*s["x"])
            torch.cuda.synchronize()
            s["graph"] = s["block"].capture(*s["x"])
    elif kind == "encoder":
        d = 64 * case["nhead"]
        T, f = case["nseq"] * case["slen"], 4 * d
        s["x"] = _normal(seed, [(T, d), (d, 3 * d), (d, d), (d, f), (f, d), (T, d)])
        s["layer"] = encoder.UnitScaledEncoderLayer(case["nseq"], case["slen"], d, case["nhead"], f, attention=case["attention"],
                                                    norm=case["norm"] or None, fused_attention=case["fused"])
        if case["norm"]:
            w1, c1, w2, c2 = _normal(seed + 1, [(d,)] * 4)
            s["ln"] = (1 + 0.1 * w1, 0.1 * c1, 1 + 0.1 * w2, 0.1 * c2)
    elif kind == "linear":
        b, m, n = case["b"], case["m"], case["n"]
        act, grad = OPERANDS[case["operand"]]
        x, w, g = _normal(seed, [(b, m), (m, n), (b, n)])
        s["x"], s["w"], s["g"] = x.to(act), w.to(act), g.to(grad)
        out = OUTPUTS[case["out"]]
        s["y"], s["dx"] = (torch.empty((b, k), dtype=out, device="cuda") for k in (n, m))
        s["dw"] = torch.empty((m, n), device="cuda")
        s["scales"], s["ws"] = L.us_scales_linear(b, m, n), L.new_workspace()
    else:
        T, d, v = case["tokens"], case["d"], case["classes"]
        x, w = _normal(seed, [(T, d), (d, v)])
        s["x"], s["w"] = x, _padded(d, v, torch.float32).copy_(w)
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        s["t"] = torch.randint(0, v, (T,), generator=gen, device="cuda", dtype=torch.int32)
        s["xq"], s["wq"] = torch.empty((T, d), dtype=E4, device="cuda"), _padded(d, v, E4)
        s["logits"], s["dlogits"] = _padded(T, v, torch.bfloat16), _padded(T, v, E5)
        s["loss"], s["dx"], s["dw"] = torch.empty(T, device="cuda"), torch.empty((T, d), dtype=torch.bfloat16, device="cuda"), _padded(d, v, torch.float32)
        s["scales"], s["ws"] = L.us_scales_linear(T, d, v), L.new_workspace()
        s["beta"] = v / math.sqrt(v - 1)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "step":
        b = s["block"]
        if c["graph"]:
            s["graph"].replay()
        else:
            b.step(*s["x"])
        return {"R": b.R, "dX": b.dX, "dW1": b.dW1, "dW2": b.dW2}
    if kind == "forward":
        return {"R": s["block"].forward(s["x"][0])}
    if kind == "encoder":
        y = s["layer"]
        out = {"dX": y.step(*s["x"], ln=s.get("ln")), "R": y.R2 if c["norm"] else y.ffn.R,
               "dWqkv": y.dWqkv, "dWo": y.dWo, "dW1": y.ffn.dW1, "dW2": y.ffn.dW2}
        if c["norm"]:
            out["dln"] = list(y.dln)
        return out
    a, bx, bw = s["scales"]
    ws = s["ws"]
    if kind == "linear":
        L.us_linear_fwd(s["x"], s["w"], a, s["y"], ws)
        L.us_linear_bwd_x(s["g"], s["w"], bx, s["dx"], ws)
        L.us_linear_bwd_w(s["x"], s["g"], bw, s["dw"], ws)
        return {"y": s["y"], "dx": s["dx"], "dw": s["dw"]}
    L.us_cast_fp8(s["x"], 1.0, s["xq"])
    L.us_cast_fp8(s["w"], 1.0, s["wq"])
    L.us_linear_fwd(s["xq"], s["wq"], a, s["logits"], ws)
    L.us_softmax_xent_fwd(s["logits"], s["t"], s["loss"])
    L.us_softmax_xent_bwd(s["logits"], s["t"], None, s["beta"], s["dlogits"])
    L.us_linear_bwd_x(s["dlogits"], s["wq"], bx, s["dx"], ws)
    L.us_linear_bwd_w(s["xq"], s["dlogits"], bw, s["dw"], ws)
    return {"logits": s["logits"], "loss": s["loss"], "dx": s["dx"], "dw": s["dw"]}


def work(case):
    """Bytes of the inputs and results of a pass (each once), and the operations of its matrix products."""
    kind = case["kind"]
    if kind == "step":          # float32 X, W1, W2, G in; 16-bit R, dX and float32 dW1, dW2 out
        T, d, f = case["tokens"], case["d"], case["f"]
        return {"bytes": 12 * T * d + 16 * d * f, "flops": 12.0 * T * d * f}
    if kind == "forward":       # float32 X and the quantised weights in, 16-bit R out
        T, d, f = case["tokens"], case["d"], case["f"]
        return {"bytes": 6 * T * d + 2 * d * f * (1 if case["operand"] == "fp8" else 2), "flops": 4.0 * T * d * f}
    if kind == "encoder":       # float32 X, G and the weights (4 d^2 + 2 d f of them) in; 16-bit R, dX and the float32 gradients out
        d = 64 * case["nhead"]
        T, w = case["nseq"] * case["slen"], 4 * d * d + 8 * d * d
        return {"bytes": 12 * T * d + 8 * w, "flops": 6.0 * T * w + 12.0 * T * case["slen"] * d}
    if kind == "linear":
        b, m, n = case["b"], case["m"], case["n"]
        e, o = 1 if case["operand"] == "fp8" else 2, {"f32": 4, "bf16": 2, "fp16": 2}.get(case["out"], 1)
        return {"bytes": e * (b * m + m * n + b * n) + o * (b * n + b * m) + 4 * m * n, "flops": 6.0 * b * m * n}
    T, d, v = case["tokens"], case["d"], case["classes"]
    return {"bytes": 6 * T * d + 8 * d * v + 2 * T * v + 8 * T, "flops": 6.0 * T * d * v}


def tolerance(case):
    """About four times the largest difference seen between this path and the same chain of products, functions and
    roundings evaluated in float64, over the listed cases and forty drawn ones.  What remains between two correct
    implementations are single codes of an intermediate or result that round the other way; an encoder layer hands
    them on through some thirty roundings, and its softmax gradient enlarges them."""
    kind = case["kind"]
    if kind == "encoder":       # seen: 2.6e-2 and 0.49
        return {"rel": 3e-2, "max": 0.99}
    if kind == "linear":        # seen: FP8 results 7e-4 and 0.11 (one code), 16-bit 2e-4 and 7.8e-3 (one ulp), float32 6.2e-6 and 2e-5
        return {"f32": {"rel": 2.5e-5, "max": 1e-4}, "e4m3": {"rel": 2.8e-3, "max": 0.45}}.get(case["out"], {"rel": 8e-4, "max": 0.032})
    if kind == "head":          # seen: 2.9e-4 and 7.8e-3
        return {"rel": 1.2e-3, "max": 0.032}
    return {"rel": 1.5e-3, "max": 0.15}     # seen: 3.7e-4 and 3.8e-2
