"""Unit-scaled Transformer encoder layer (self-attention block + FFN block), forward and backward,
as a sequence of libunitscale calls.  A driver only: buffers and call order; all arithmetic runs
in the library's kernels.

Layer (no layer norm; fixed(tau) residuals, section "Weighted addition"):
    QKV = alpha_qkv q(X) q(Wqkv)                          FP8 GEMM, 16-bit output [T x 3d]
    S   = alpha_s Q_h K_h^T   per (sequence, head)        batched, 16-bit operands, alpha_s = 1/sqrt(d_head)
    P   = s softmax(S)                                    scaled softmax (table row "softmax"), s = sequence length
    C   = alpha_c P V_h                                   batched, alpha_c = s^-1/2, stored as E4M3
    R1  = sqrt(1-tau) X + sqrt(tau) alpha_o C q(Wo)       FP8 GEMM + residual epilogue
    R2  = FFN block on R1                                 see ffn.py
Backward from G = dL/dR2: the FFN block's backward gives g1 = dL/dR1, then
    dC  = beta_o q(g1) q(Wo)^T ; dWo = beta_w C^T q(g1)
    dP  = beta_P dC_h V_h^T ; dV = beta_V P^T dC_h        batched
    dS  = s softmax_grad(P, dP)
    dQ  = beta_Q dS K_h ; dK = beta_K dS^T Q_h            batched
    dX  = sqrt(1-tau) g1 + sqrt(tau) beta_qkv q(dQKV) q(Wqkv)^T ; dWqkv = beta_w q(X)^T q(dQKV)
Scale factors are the unconstrained table values (alpha = fan_in^-1/2, beta_X = fan_out^-1/2,
beta_W = batch^-1/2 with the batch of an attention matmul = its sequence length).

attention = "bf16" / "fp16": the attention matmuls take 16-bit operands.  attention = "fp8": they take
FP8 operands like the projections (section "Experiments": all matmul inputs are quantised): the QKV
GEMM writes Q, K, V as E4M3, the softmax writes P as E4M3, the gradients dC and dS are written as E5M2
and the batched GEMMs write dQ, dK, dV straight into the E5M2 operand of the QKV backward GEMMs (one
cast launch fewer); S and dP, which feed no matmul, stay in BF16.
"""
from __future__ import annotations


import torch

from . import ffn as F
from . import lib as L

E4, E5 = torch.float8_e4m3fn, torch.float8_e5m2


def backward_in_one_launch(problems: int, slen: int, fp8: bool) -> bool:
    """Whether the backward pass of fused attention over `problems` (sequence, head) pairs goes out as one launch instead of three.

    Up to 128 keys a CTA holds a problem, and one launch is faster at any size (8192 tokens of 16 heads, 16 / 64 / 128 keys: the layer
    takes 131 / 40 / 27 us less).  Up to 256 a cluster of two does, 74 of which run at once; beyond, one of four, 33 at once, that walks
    the problem's query tiles one after another, while the three launches give each tile to one of 148 CTAs.  So the line depends on the
    waves of both, and on the keys that a cluster's last CTA has.  Layers of 2 to 6 heads, us that one launch adds (a list: problems):
      144 keys, 16-bit, 12 / 36 / 40 / 80 / 150 / 300: +1.1 -0.7 -1.3 -0.5 +0.4 +4.4; 192: +0.7 +0.5 -2.0 -0.4 0 +0.5 (12 heads, 252:
      +1.3); 208: 0 -0.2 -2.5 -2.2 -2.9 -4.4; 256: 0 -0.7 -2.6 -2.0 -2.8 -9.2
      144 keys, FP8: +0.8 -0.8 -1.6 -2.0 -2.5 -3.7; 256: 0 0 -1.5 -2.5 -3.5 -5.8
      336 keys, 16-bit, 8 / 20 / 32 / 36 / 64 / 96 / 192 / 256: +0.7 -0.7 -1.8 +6.9 -1.9 +5.2 +10.5 +13.8; 448: +1.4 -0.7 -1.7 +8.1 -0.7 -3.0 -5.9 +3.2;
      480: +0.7 -1.4 -3.1 +7.8 -3.4 -7.8 -15.3 -8.6; 512: +0.8 -1.0 -3.7 +6.3 -5.5 -11.0 -22.4 -16.3
      336 keys, FP8: -0.2 -1.3 -1.9 +5.0 -0.5 +5.1 +15.8 +19.9; 448: +0.5 -1.2 -1.7 +7.6 -1.1 -0.4 +2.4 +11.5; 512: +0.7 -0.6 -1.6 +7.0 -1.8 -2.2 -1.4 +4.2
      272 to 320 keys: within 1.4 up to 33 problems, +0.2 to +23 beyond"""
    if slen <= 128:
        return True
    if slen <= 256:
        return problems >= 37 and (fp8 or slen >= 208 or problems <= 80)
    waves, waves_of_three = -(-problems // 33), -(-problems * -(-slen // 128) // 148)
    if slen < 336 or problems < 20:
        return False
    if fp8:
        return waves <= min(3, waves_of_three)
    return waves * (0.8 if slen >= 480 else 0.92 if slen >= 448 else 1.0) <= waves_of_three


class UnitScaledEncoderLayer:
    def __init__(self, nseq: int, slen: int, d: int, nhead: int, d_ff: int, tau: float = 0.5,
                 attention: str = "bf16", norm: str | None = None, eps: float = 1e-5, device="cuda",
                 fused_attention: bool = False):
        assert d % nhead == 0 and norm in (None, "post")
        self.attention, self.norm, self.eps = attention, norm, eps
        # fused_attention: scores, scaled softmax and context of the forward pass as one us_attention_fwd launch, and the
        # whole backward pass as one us_attention_bwd_all launch, or dP, the softmax gradient and dQ as one us_attention_bwd
        # launch (heads of 64, at most 512 tokens per sequence; 16-bit or FP8 attention operands); the scores and the
        # gradient dP are then never stored
        self.fused_attention = fused_attention
        if fused_attention and not (d // nhead == 64 and slen <= 512):
            raise ValueError("fused attention needs heads of 64 and sequences of at most 512 tokens")
        if attention == "fp8":
            act_dt, grad_dt, wide_dt = E4, E5, torch.bfloat16
        else:
            act_dt = grad_dt = wide_dt = {"bf16": torch.bfloat16, "fp16": torch.float16}[attention]
        self.nseq, self.slen, self.d, self.nhead, self.hd, self.d_ff, self.tau = nseq, slen, d, nhead, d // nhead, d_ff, tau
        T = self.T = nseq * slen
        e = lambda r, c, dt: torch.empty((r, c), dtype=dt, device=device)
        self.Xq, self.Wqkv_q, self.Wo_q = e(T, d, E4), e(d, 3 * d, E4), e(d, d, E4)
        self.QKV = e(T, 3 * d, act_dt)
        self.S = None if fused_attention else e(nseq * nhead * slen, slen, wide_dt)
        self.P = e(nseq * nhead * slen, slen, act_dt)
        self.Cq = e(T, d, E4)
        self.R1 = e(T, d, torch.bfloat16)
        self.ffn = F.UnitScaledFFN(T, d, d_ff, scales=F.FFNScales.unit(T, d, d_ff, tau), device=device)
        self.g1q = e(T, d, E5)
        self.dC = e(T, d, grad_dt)
        self.dP = None if fused_attention else e(nseq * nhead * slen, slen, wide_dt)
        self.dS = e(nseq * nhead * slen, slen, grad_dt)
        self.dQKVq = e(T, 3 * d, E5)
        # dQ, dK, dV are consumed only as the E5M2 operand of the QKV projection's backward GEMMs: with FP8 attention
        # operands, and with the fused attention kernels, their producers write that format directly (no cast launch)
        self.dQKV = self.dQKVq if (attention == "fp8" or fused_attention) else e(T, 3 * d, grad_dt)
        self.dX = e(T, d, torch.bfloat16)
        self.dWqkv, self.dWo = e(d, 3 * d, torch.float32), e(d, d, torch.float32)
        self.ws = L.new_workspace(device)
        self._plan = self._events = None
        if norm == "post":
            # post-norm (appendix "Model architectures"): a scaled layer norm after each residual sum
            self.U1, self.R2 = e(T, d, torch.bfloat16), e(T, d, torch.bfloat16)
            self.dU1, self.dU2 = e(T, d, torch.bfloat16), e(T, d, torch.bfloat16)
            self.dln = [torch.empty(d, dtype=torch.float32, device=device) for _ in range(4)]      # dw1, dc1, dw2, dc2
            self.ln_ws = torch.empty(max(16, L.us_layer_norm_bwd_workspace_bytes(T, d)), dtype=torch.uint8, device=device)
            self.beta_ln = L.us_scales_linear(T, 1, 1)[2]          # b^-1/2 with b = all tokens
        self.c_skip, self.c_branch = L.us_scales_residual(tau)
        s, hd = slen, self.hd
        a_qkv, b_qkv, b_w = L.us_scales_linear(T, d, 3 * d)
        a_o, b_o, _ = L.us_scales_linear(T, d, d)
        self.sc = dict(alpha_qkv=a_qkv, beta_qkv=b_qkv, alpha_o=a_o, beta_o=b_o, beta_w=b_w, **L.us_scales_attention(s, hd))
        qkv = (slen * 3 * d, hd)          # (outer, inner) strides of a head slice of a [T x 3d] matrix
        sq = (nhead * slen * slen, slen * slen)
        td = (slen * d, hd)               # head slice of a [T x d] matrix
        n = (nseq, nhead)
        self.bt = dict(scores=L.batch(n, qkv, qkv, sq), ctx=L.batch(n, sq, qkv, td), dP=L.batch(n, td, qkv, sq),
                       dV=L.batch(n, sq, td, qkv), dQ=L.batch(n, sq, qkv, qkv), dK=L.batch(n, sq, qkv, qkv))
        # fused cast, attention forward, FFN forward + backward, attention backward (one cast fewer with FP8 attention)
        self._launches = 1 + (3 if fused_attention else 5) + 7 + ((10 if (attention == "fp8" or fused_attention) else 11) - (2 if fused_attention else 0)) + (7 if norm == "post" else 0)
        self.bt_fused = L.attention_batch(n, qkv, qkv, qkv, td, sq)
        self.bt_fused_bwd = L.attention_bwd_batch(n, td, sq, qkv, qkv, sq, qkv)
        self.bt_fused_all = L.attention_bwd_all_batch(n, td, sq, qkv, qkv, qkv, sq, qkv, qkv, qkv)
        self._whole = backward_in_one_launch(nseq * nhead, slen, attention == "fp8")

    @property
    def whole_bwd(self) -> bool:
        """Whether the backward pass of attention is one launch."""
        return self.fused_attention and self._whole

    @property
    def launches_per_step(self) -> int:
        """Library operations of one step with every GEMM of the layer itself counted (the FFN block's six GEMMs as its
        gemm_launches, without layer norms; the backward pass of fused attention as three operations: dQ, dK, dV).  The
        gradient GEMMs of a projection go out together: kernel_launches is the number of kernels."""
        return self._launches - (6 - self.ffn.gemm_launches if self.norm is None else 0)

    @property
    def kernel_launches(self) -> int:
        """Kernel launches of one step: launches_per_step with the two gradient GEMMs of a projection, with layer norms the three
        GEMMs that end the FFN block's backward pass, and the fused backward pass of attention as the launches they make, and
        less the casts that their tensors' producers make."""
        together = sum(2 - L.us_linear_group_launches(calls) for calls in (self._out_grads(), self._qkv_grads()))
        if self.norm is not None and self.ffn.grouped:
            together += 3 - self.ffn._group_launches(forward=False)
        return self.launches_per_step - together - (2 if self.whole_bwd else 0) - (2 if self.norm is None else 3)

    def _out_grads(self):
        """Gradient GEMMs of the output projection."""
        sc = self.sc
        return [L.linear_call(L.US_OP_BWD_W, self.Cq, self.g1q, sc["beta_w"], self.dWo), L.linear_call(L.US_OP_BWD_X, self.g1q, self.Wo_q, sc["beta_o"], self.dC)]

    def _qkv_grads(self, ep=None):
        """Gradient GEMMs of the query, key and value projections."""
        sc = self.sc
        return [L.linear_call(L.US_OP_BWD_W, self.Xq, self.dQKVq, sc["beta_w"], self.dWqkv),
                L.linear_call(L.US_OP_BWD_X, self.dQKVq, self.Wqkv_q, sc["beta_qkv"], self.dX, ep)]

    def _heads(self, M, which):
        """Problem (0, 0) of a [T x 3d] matrix: rows of the first sequence, columns of head 0 of Q / K / V."""
        o = which * self.d
        return M[: self.slen, o:o + self.hd]

    # ---- a step as calls laid out once over the layer's buffers (L.Plan), the same ones as _step_each, as (where, call) pairs
    MAIN, SIDE, JOIN = L.Plan.MAIN, L.Plan.SIDE, L.Plan.JOIN

    def _owned(self):
        own = (self.Xq, self.Wqkv_q, self.Wo_q, self.QKV, self.P, self.Cq, self.R1, self.g1q, self.dC, self.dS, self.dQKVq, self.dQKV,
               self.dX, self.dWqkv, self.dWo, self.ws) + self.ffn._owned()
        if not self.fused_attention:
            own += (self.S, self.dP)
        if self.norm == "post":
            own += (self.U1, self.R2, self.dU1, self.dU2, self.ln_ws, *self.dln)
        return own

    def _state(self):
        return (*self.sc.values(), self.c_skip, self.c_branch, self.eps, self.beta_ln if self.norm else 0.0) + self.ffn._state()

    def _lay_out(self, p):
        sc, ws, s, f = self.sc, self.ws, self.slen, self.ffn
        post, fused = self.norm == "post", self.fused_attention
        coef = (self.c_skip, self.c_branch)
        MAIN = self.MAIN

        # a tensor that is the operand of a matmul too leaves its producer in FP8 as well
        def norm_bwd(X, w, G, dX, dXq, dw, dc):
            g = p.slot(G) if isinstance(G, str) else p.mat(G)
            return L.Call("us_layer_norm_bwd_cast", p.mat(X), p.slot(w), g, self.eps, 1.0, self.beta_ln, p.mat(dX), p.mat(dXq), L._vec(dw), L._vec(dc),
                          self.ln_ws.data_ptr(), self.ln_ws.numel())

        # the first pass issues each call as it is laid out, so nothing is made before the call that needs it
        yield MAIN, p.cast_multi(["Wqkv", "Wo", "X", "W1", "W2"] + ([] if post else ["G"]),
                                 [self.Wqkv_q, self.Wo_q, self.Xq, f.W1q, f.W2q] + ([] if post else [f.Gq]))
        yield MAIN, p.linear("us_linear_fwd", self.Xq, self.Wqkv_q, sc["alpha_qkv"], self.QKV, ws)
        Q, K, V = (self._heads(self.QKV, i) for i in range(3))
        P, C_h = self.P[:s], self.Cq[:s, : self.hd]
        tail = (ws.data_ptr(), ws.numel())
        if fused:
            yield MAIN, L.Call("us_attention_fwd", p.mat(Q), p.mat(K), p.mat(V), sc["alpha_s"], sc["sm"], sc["alpha_c"], p.mat(C_h), p.mat(P),
                               self.bt_fused, *tail)
        else:
            yield MAIN, p.batched("us_linear_bwd_x_batched", Q, K, sc["alpha_s"], self.S[:s], self.bt["scores"], ws)
            yield MAIN, L.Call("us_softmax_fwd", p.mat(self.S), sc["sm"], p.mat(self.P))
            yield MAIN, p.batched("us_linear_fwd_batched", P, V, sc["alpha_c"], C_h, self.bt["ctx"], ws)
        if post:
            yield MAIN, p.linear("us_linear_fwd", self.Cq, self.Wo_q, sc["alpha_o"], self.U1, ws, p.residual("X", coef))
            yield MAIN, L.Call("us_layer_norm_fwd_cast", p.mat(self.U1), p.slot("w1"), p.slot("c1"), self.eps, p.mat(self.R1), p.mat(f.Xq))
            for c in f.plan_forward(p, self.R1, cast_x=False):
                yield MAIN, c
            yield MAIN, L.Call("us_layer_norm_fwd", p.mat(f.R), p.slot("w2"), p.slot("c2"), self.eps, p.mat(self.R2))
            yield MAIN, norm_bwd(f.R, "w2", "G", self.dU2, f.Gq, self.dln[2], self.dln[3])
            for c in f.plan_backward(p, self.dU2, cast_g=False):
                yield MAIN, c
            yield MAIN, norm_bwd(self.U1, "w1", f.dX, self.dU1, self.g1q, self.dln[0], self.dln[1])
            g1 = self.dU1
        else:
            yield MAIN, L.Call("us_linear_fwd_cast", p.mat(self.Cq), p.mat(self.Wo_q), sc["alpha_o"], p.residual("X", coef), p.mat(self.R1),
                               p.mat(f.Xq), *tail)
            for c in f.plan_gemms(p, self.R1, "G", self.g1q):
                yield MAIN, c
            g1 = f.dX
        yield MAIN, p.group([(L.US_OP_BWD_W, self.Cq, self.g1q, sc["beta_w"], self.dWo, None, None),
                             (L.US_OP_BWD_X, self.g1q, self.Wo_q, sc["beta_o"], self.dC, None, None)], ws)
        dQ, dK, dV = (self._heads(self.dQKV, i) for i in range(3))
        dS, dC_h = self.dS[:s], self.dC[:s, : self.hd]
        if self.whole_bwd:
            # dS is read by no later launch; it is stored (7 us of 8192 tokens of 16 heads and 512 keys at 16 bits) because self.dS holds
            # it after a step, as with three launches
            yield MAIN, L.Call("us_attention_bwd_all", *(p.mat(t) for t in (dC_h, P, Q, K, V)), sc["beta_P"], sc["sm"], sc["sm"], sc["beta_Q"],
                               sc["beta_K"], sc["beta_V"], *(p.mat(t) for t in (dS, dQ, dK, dV)), self.bt_fused_all, *tail)
        else:
            yield self.SIDE, p.batched("us_linear_bwd_w_batched", P, dC_h, sc["beta_V"], dV, self.bt["dV"], ws)
            gemm_dk = p.batched("us_linear_bwd_w_batched", dS, Q, sc["beta_K"], dK, self.bt["dK"], ws)
            if fused:
                yield MAIN, L.Call("us_attention_bwd", p.mat(dC_h), p.mat(P), p.mat(K), p.mat(V), sc["beta_P"], sc["sm"], sc["sm"], sc["beta_Q"],
                                   p.mat(dS), p.mat(dQ), self.bt_fused_bwd, *tail)
                yield self.SIDE, gemm_dk
            else:
                yield MAIN, p.batched("us_linear_bwd_x_batched", dC_h, V, sc["beta_P"], self.dP[:s], self.bt["dP"], ws)
                yield MAIN, L.Call("us_softmax_bwd", p.mat(self.P), p.mat(self.dP), sc["sm"], sc["sm"], p.mat(self.dS))
                yield self.SIDE, gemm_dk
                yield MAIN, p.batched("us_linear_fwd_batched", dS, K, sc["beta_Q"], dQ, self.bt["dQ"], ws)
            yield self.JOIN, None                                   # dQ, dK, dV all written
        if self.dQKV is not self.dQKVq:
            yield MAIN, L.Call("us_cast_fp8", p.mat(self.dQKV), 1.0, p.mat(self.dQKVq))
        yield MAIN, p.group([(L.US_OP_BWD_W, self.Xq, self.dQKVq, sc["beta_w"], self.dWqkv, None, None),
                             (L.US_OP_BWD_X, self.dQKVq, self.Wqkv_q, sc["beta_qkv"], self.dX, g1, coef)], ws)

    def __getstate__(self):
        """A copy has buffers of its own: its plan is laid out, and its events are made, by its first step."""
        return {**self.__dict__, "_plan": None, "_events": None}

    def _run(self, stream, **inputs):
        owned, state = self._owned(), self._state()
        p = self._plan
        if p is None or not p.same(owned, state):
            p = self._plan = L.Plan(owned, state)
        if self.whole_bwd or not (stream is None and self.ffn.concurrent):
            p.issue(self._lay_out, inputs, L._stream(stream))
            return
        cur = torch.cuda.current_stream()
        if self._events is None:
            self._events = torch.cuda.Event(), torch.cuda.Event()
            for e in self._events:
                e.record(cur)                                       # an event has a handle once it has been recorded
        p.issue(self._lay_out, inputs, cur.cuda_stream, (self.ffn._side_streams()[0], *self._events))

    def step(self, X, Wqkv, Wo, W1, W2, G, stream=None, ln=None):
        """One forward + backward pass.  G is the gradient of the layer output; with norm = "post",
        ln = (w1, c1, w2, c2) are the weights and biases of the two layer norms ([d] each)."""
        if self.ffn.grouped and self.ffn.fused_hidden:
            norm = dict(zip(("w1", "c1", "w2", "c2"), (t.view(1, -1) for t in ln))) if self.norm == "post" else {}
            self._run(stream, X=X, Wqkv=Wqkv, Wo=Wo, W1=W1, W2=W2, G=G, **norm)
            return self.dX
        return self._step_each(X, Wqkv, Wo, W1, W2, G, stream, ln)

    def _step_each(self, X, Wqkv, Wo, W1, W2, G, stream, ln):
        """step() call by call, for an FFN block whose grouped forms are switched off."""
        sc, ws, s = self.sc, self.ws, self.slen
        post = self.norm == "post"
        # ---- forward
        f = self.ffn
        # every tensor that is known when the step starts goes to FP8 in one launch (with post-norm the FFN
        # block's incoming gradient is produced by the second norm's backward pass and is cast there)
        dsts = [self.Wqkv_q, self.Wo_q, self.Xq, f.W1q, f.W2q] + ([] if post else [f.Gq])
        (L.us_cast_multi_pitched if L._padded(dsts) else L.us_cast_fp8_multi)([Wqkv, Wo, X, W1, W2] + ([] if post else [G]), [1.0] * len(dsts), dsts, stream)
        L.us_linear_fwd(self.Xq, self.Wqkv_q, sc["alpha_qkv"], self.QKV, ws, None, stream)
        Q, K, V = (self._heads(self.QKV, i) for i in range(3))
        if self.fused_attention:
            L.us_attention_fwd(Q, K, V, sc["alpha_s"], sc["sm"], sc["alpha_c"], self.Cq[:s, : self.hd], self.P[:s],
                               self.bt_fused, ws, stream)
        else:
            L.us_linear_bwd_x_batched(Q, K, sc["alpha_s"], self.S[:s], self.bt["scores"], ws, stream)
            L.us_softmax_fwd(self.S, sc["sm"], self.P, stream)
            L.us_linear_fwd_batched(self.P[:s], V, sc["alpha_c"], self.Cq[:s, : self.hd], self.bt["ctx"], ws, stream)
        ep = L.epilogue(skip=X, skip_coef=self.c_skip, out_coef=self.c_branch)
        L.us_linear_fwd(self.Cq, self.Wo_q, sc["alpha_o"], self.U1 if post else self.R1, ws, ep, stream)
        if post:
            L.us_layer_norm_fwd(self.U1, ln[0], ln[1], self.eps, self.R1, stream)
        if post or not f.grouped:
            f.forward(self.R1, stream)
        # ---- backward
        if post:
            L.us_layer_norm_fwd(f.R, ln[2], ln[3], self.eps, self.R2, stream)
            L.us_layer_norm_bwd(f.R, ln[2], G, self.eps, 1.0, self.beta_ln, self.dU2, self.dln[2], self.dln[3], self.ln_ws, stream)
            f.backward(self.dU2, stream)                            # f.dX = dL/dR1
            L.us_layer_norm_bwd(self.U1, ln[0], f.dX, self.eps, 1.0, self.beta_ln, self.dU1, self.dln[0], self.dln[1], self.ln_ws, stream)
            g1 = self.dU1
        elif f.grouped:
            # G is known from the start, so the whole FFN block goes out as a cast of its input and three GEMM launches
            f._cast(self.R1, f.Xq, stream)
            f.step_from_casts(self.R1, G, stream)                   # f.R = layer output, f.dX = dL/dR1
            g1 = f.dX
        else:
            f.backward(G, stream, cast_g=False)                     # f.dX = dL/dR1
            g1 = f.dX
        # The two gradient GEMMs of a projection are independent of one another and go out as one launch, the weight
        # gradient's long contractions dealt out first.  One GEMM of each attention pair depends only on tensors that
        # exist already; with no explicit stream it goes to a side stream (a parallel branch under graph capture).
        par = stream is None and f.concurrent
        cur = torch.cuda.current_stream() if par else stream
        side = f._side_streams()[0] if par else stream

        def beside(fn):
            """Run fn on the side stream once everything issued so far on the main stream is done."""
            if par:
                ev = torch.cuda.Event()
                ev.record(cur)
                side.wait_event(ev)
            fn(side)

        L.us_cast_fp8(g1, 1.0, self.g1q, cur)
        L.linear_together(self._out_grads(), ws, cur)
        dC_h = self.dC[:s, : self.hd]
        if self.whole_bwd:
            L.us_attention_bwd_all(dC_h, self.P[:s], Q, K, V, sc["beta_P"], sc["sm"], sc["sm"], sc["beta_Q"], sc["beta_K"], sc["beta_V"],
                                   self.dS[:s], *(self._heads(self.dQKV, i) for i in range(3)), self.bt_fused_all, ws, cur)
        else:
            beside(lambda st: L.us_linear_bwd_w_batched(self.P[:s], dC_h, sc["beta_V"], self._heads(self.dQKV, 2), self.bt["dV"], ws, st))
            gemm_dk = lambda st: L.us_linear_bwd_w_batched(self.dS[:s], Q, sc["beta_K"], self._heads(self.dQKV, 1), self.bt["dK"], ws, st)
            if self.fused_attention:
                L.us_attention_bwd(dC_h, self.P[:s], K, V, sc["beta_P"], sc["sm"], sc["sm"], sc["beta_Q"], self.dS[:s],
                                   self._heads(self.dQKV, 0), self.bt_fused_bwd, ws, cur)
                beside(gemm_dk)
            else:
                L.us_linear_bwd_x_batched(dC_h, V, sc["beta_P"], self.dP[:s], self.bt["dP"], ws, cur)
                L.us_softmax_bwd(self.P, self.dP, sc["sm"], sc["sm"], self.dS, cur)
                beside(gemm_dk)
                L.us_linear_fwd_batched(self.dS[:s], K, sc["beta_Q"], self._heads(self.dQKV, 0), self.bt["dQ"], ws, cur)
        if par:
            cur.wait_stream(side)                                   # dQ, dK, dV all written
        if self.dQKV is not self.dQKVq:
            L.us_cast_fp8(self.dQKV, 1.0, self.dQKVq, cur)
        ep = L.epilogue(skip=g1, skip_coef=self.c_skip, out_coef=self.c_branch)
        L.linear_together(self._qkv_grads(ep), ws, cur)
        return self.dX

    def check(self) -> None:
        for ws in (self.ws, self.ffn.ws):
            st = L.us_workspace_status(ws)
            if st != L.US_OK:
                raise L.UnitScaleError("UnitScaledEncoderLayer", st)

    def flops(self) -> float:
        T, d, f, s, hd = self.T, self.d, self.d_ff, self.slen, self.hd
        proj = 6.0 * T * d * 3 * d + 6.0 * T * d * d
        att = 2 * 6.0 * (self.nseq * self.nhead) * s * s * hd
        return proj + att + 12.0 * T * d * f
