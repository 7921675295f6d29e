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


# ---- the same results in 64 bits: the chain of products, functions and storage formats, in plain torch

_BF, _C = torch.bfloat16, math.sqrt(0.5)      # both residual coefficients (tau = 1/2)


def _q(v, dtype):
    """The values of v in a storage format (FP8 casts saturate)."""
    most = {E4: 448.0, E5: 57344.0}.get(dtype)
    return (v if most is None else v.clamp(-most, most)).to(dtype).double()


def _phi_pdf(z):
    return 0.5 * torch.erfc(-z * math.sqrt(0.5)), torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)


def _ffn64(X, W1, W2, G, act, grad):
    T, (d, f) = X.shape[0], W1.shape
    Xq, W1q, W2q = _q(X, act), _q(W1, act), _q(W2, act)
    H = d ** -0.5 * (Xq @ W1q)
    A = _q(1.7009262 * H * _phi_pdf(H)[0], act)
    R = _q(_C * X + _C * f ** -0.5 * (A @ W2q), _BF)
    if G is None:
        return {"R": R}
    H, Gq = _q(H, _BF), _q(G, grad)
    P, p = _phi_pdf(H)
    dH = _q(1.4811144 * (P + H * p) * d ** -0.5 * (Gq @ W2q.T), grad)
    return {"R": R, "dX": _q(_C * G + _C * f ** -0.5 * (dH @ W1q.T), _BF), "dW1": T ** -0.5 * (Xq.T @ dH), "dW2": T ** -0.5 * (A.T @ Gq)}


def _norm64(U, w, c):
    m = U.mean(1, keepdim=True)
    s = ((U - m).square().mean(1, keepdim=True) + 1e-5).sqrt()
    return _q((U - m) / s * w + c, _BF), (U - m) / s, s


def _norm_bwd64(xh, s, w, g):
    gw, b = g * w, g.shape[0] ** -0.5
    dx = (gw - gw.mean(1, keepdim=True) - xh * (gw * xh).mean(1, keepdim=True)) / s
    return _q(dx, _BF), b * (g * xh).sum(0), b * g.sum(0)


def _encoder64(case, X, Wqkv, Wo, W1, W2, G, ln):
    ns, s, nh, fused = case["nseq"], case["slen"], case["nhead"], case["fused"]
    T, d, hd = X.shape[0], X.shape[1], 64
    act, grad, wide = (E4, E5, _BF) if case["attention"] == "fp8" else (OUTPUTS[case["attention"]],) * 3
    mid = (lambda v, dt: v) if fused else _q       # the fused kernels keep scores and their gradient unrounded

    def heads(M):
        return M.reshape(ns, s, nh, hd).transpose(1, 2)

    def rows(H):
        return H.transpose(1, 2).reshape(T, nh * hd)
    Xq, Wqkv_q, Wo_q = _q(X, E4), _q(Wqkv, E4), _q(Wo, E4)
    Q, K, V = (heads(m) for m in _q(d ** -0.5 * (Xq @ Wqkv_q), act).split(d, 1))
    P = _q(s * torch.softmax(mid(hd ** -0.5 * (Q @ K.transpose(2, 3)), wide), -1), act)
    C = _q(rows(s ** -0.5 * (P @ V)), E4)
    U1 = R1 = _q(_C * X + _C * d ** -0.5 * (C @ Wo_q), _BF)
    if ln:
        R1, xh1, s1 = _norm64(U1, ln[0], ln[1])
        F = _ffn64(R1, W1, W2, None, E4, E5)["R"]
        R, xh2, s2 = _norm64(F, ln[2], ln[3])
        g2, dw2, dc2 = _norm_bwd64(xh2, s2, ln[2], G)
        f = _ffn64(R1, W1, W2, g2, E4, E5)
        g1, dw1, dc1 = _norm_bwd64(xh1, s1, ln[0], f["dX"])
    else:
        f = _ffn64(R1, W1, W2, G, E4, E5)
        R, g1 = f["R"], f["dX"]
    g1q = _q(g1, E5)
    dC = heads(_q(d ** -0.5 * (g1q @ Wo_q.T), grad))
    dP = mid(hd ** -0.5 * (dC @ V.transpose(2, 3)), wide)
    p = P / s
    dS = _q(s * p * (dP - (p * dP).sum(-1, keepdim=True)), grad)
    dQKV = torch.cat([rows(hd ** -0.5 * (dS @ K)), rows(hd ** -0.5 * (dS.transpose(2, 3) @ Q)), rows(s ** -0.5 * (P.transpose(2, 3) @ dC))], 1)
    dQKV = _q(dQKV if fused else _q(dQKV, grad), E5)
    out = {"dX": _q(_C * g1 + _C * (3 * d) ** -0.5 * (dQKV @ Wqkv_q.T), _BF), "R": R, "dWqkv": T ** -0.5 * (Xq.T @ dQKV),
           "dWo": T ** -0.5 * (C.T @ g1q), "dW1": f["dW1"], "dW2": f["dW2"]}
    if ln:
        out["dln"] = [dw1, dc1, dw2, dc2]
    return out


def exact(case, seed):
    """What `run` returns for these inputs, computed in float64 with the path's storage formats between the steps."""
    kind = case["kind"]
    s = prepare(dict(case, graph=False), seed)
    if kind in ("step", "forward"):
        X, W1, W2, G = (t.double() for t in s["x"])
        return _ffn64(X, W1, W2, G if kind == "step" else None, *OPERANDS[case["operand"]])
    if kind == "encoder":
        return _encoder64(case, *(t.double() for t in s["x"]), [v.double() for v in s["ln"]] if "ln" in s else None)
    if kind == "linear":
        b, m, n = case["b"], case["m"], case["n"]
        x, w, g = (s[k].double() for k in "xwg")
        out = OUTPUTS[case["out"]]
        return {"y": _q(m ** -0.5 * (x @ w), out), "dx": _q(n ** -0.5 * (g @ w.T), out), "dw": b ** -0.5 * (x.T @ g)}
    T, d, v = case["tokens"], case["d"], case["classes"]
    xq, wq, t = _q(s["x"], E4), _q(s["w"], E4), s["t"].long()[:, None]
    logits = _q(d ** -0.5 * (xq @ wq), _BF)
    logp = torch.log_softmax(logits, 1)
    g = -logp.exp()
    g.scatter_add_(1, t, torch.ones_like(t, dtype=torch.float64))
    g = _q(s["beta"] * g, E5)
    return {"logits": logits, "loss": logp.gather(1, t)[:, 0], "dx": _q(v ** -0.5 * (g @ wq.T), _BF), "dw": T ** -0.5 * (xq.T @ g)}
