"""The chained unit-scaled FFN block (forward + backward) against the oracle's chain."""
import numpy as np
import pytest
import torch

from oracle import formats as F
from oracle import ops as O
from tests import util as U

pytestmark = pytest.mark.gpu
TOL = 2e-3


def _mods():
    from paper_2303_11257_b200 import ffn, lib, synth
    return ffn, lib, synth


def _run(shape, operand, seed=0, sigma_x=1.0, io="bf16"):
    ffn, L, synth = _mods()
    X, W1, W2, G = synth.ffn_tensors(shape, seed, sigma_x)
    blk = ffn.UnitScaledFFN(shape.tokens, shape.d_model, shape.d_ff, operand=operand,
                            io_dtype=U.TORCH_OF[io], keep_h=True)
    dev = [torch.from_numpy(t).cuda() for t in (X, W1, W2, G)]
    blk.step(*dev)
    blk.check()
    return blk, (X, W1, W2, G)


def _oracle(shape, tensors, operand, io="bf16"):
    sc = O.FFNScales.unconstrained(shape.tokens, shape.d_model, shape.d_ff)
    return O.ffn_block(*tensors, sc, operand=operand, io_dtype=io)


def _compare_chain(blk, r, tensors, operand, rows=None, weights=True):
    """Stage-by-stage comparison.  Each GEMM is checked against the oracle's chain at 2e-3; where an
    upstream FP8 cast legitimately landed on the neighbouring code (a near-tie decided by float32
    vs float64 arithmetic, allowed by the one-code tolerance), the exact effect of that flip on the
    downstream matmul, |delta| @ |other operand| times the scales, is added to the tolerance."""
    sc = blk.sc
    act = "e4m3" if operand == "fp8" else operand
    grad = "e5m2" if operand == "fp8" else operand
    sel = (lambda t: t) if rows is None else (lambda t: t[torch.from_numpy(rows).cuda()])
    c_branch = float(np.float32(np.sqrt(sc.tau)))
    U.assert_close_stored(sel(blk.H), r.H, "bf16", TOL, "H")
    # A one-ulp difference in the stored 16-bit H (rare) moves gelu'(s H) by at most
    # max|gelu''| * s * |delta H| with max|gelu''| = 2 phi(0) < 0.8, hence dH by the bound below.
    dHs = np.abs(U.host_values(sel(blk.H)) - r.H)
    h_allow = 1.01 * sc.beta_g * sc.s_in ** 2 * 0.8 * dHs * np.abs(r.dA)
    if operand == "fp8":
        dA = U.code_deltas(sel(blk.Aq), r.Aq_codes, act)
        dH = U.code_deltas(sel(blk.dHq), r.dHq_codes, grad, extra=h_allow)
    else:   # 16-bit operands: values within an ulp; the actual differences are the deltas
        dA = U.host_values(sel(blk.Aq)) - r.Aq
        dH = U.host_values(sel(blk.dHq)) - r.dHq
        assert np.all(np.abs(dA) <= TOL + U.ulp_of(r.Aq, act))
        assert np.all(np.abs(dH) <= TOL + U.ulp_of(r.dHq, grad) + h_allow)
    U.assert_close_stored(sel(blk.R), r.R, "bf16", TOL + c_branch * sc.alpha2 * U.propagated(dA, r.W2q, "a"), "R")
    U.assert_close_stored(sel(blk.dX), r.dX, "bf16", TOL + c_branch * sc.beta_x1 * U.propagated(dH, r.W1q.T, "a"), "dX")
    if weights:
        U.assert_close_stored(blk.dW2, r.dW2, "f32", TOL + sc.beta_w * U.propagated(dA.T, r.Gq, "a"), "dW2")
        U.assert_close_stored(blk.dW1, r.dW1, "f32", TOL + sc.beta_w * U.propagated(r.Xq.T, dH, "b"), "dW1")


@pytest.mark.parametrize("shape_name", ["FFN_SMALL", "FFN_RAGGED"])
@pytest.mark.parametrize("operand", ["fp8", "bf16", "fp16"])
def test_ffn_block_full_compare(shape_name, operand):
    ffn, L, synth = _mods()
    shape = getattr(synth, shape_name)
    blk, tensors = _run(shape, operand)
    r = _oracle(shape, tensors, operand)
    act = "e4m3" if operand == "fp8" else operand
    grad = "e5m2" if operand == "fp8" else operand
    # casts of the same float32 values: bit-exact
    assert np.array_equal(U.codes_of(blk.Xq), F.quantise_codes(tensors[0], F.FORMATS[act]))
    assert np.array_equal(U.codes_of(blk.W1q), F.quantise_codes(tensors[1], F.FORMATS[act]))
    assert np.array_equal(U.codes_of(blk.Gq), F.quantise_codes(tensors[3], F.FORMATS[grad]))
    _compare_chain(blk, r, tensors, operand)


@pytest.fixture(scope="module")
def bert_large_fp8():
    ffn, L, synth = _mods()
    shape = synth.FFN_BERT_LARGE
    blk, tensors = _run(shape, "fp8", seed=0)
    return shape, blk, tensors


def test_ffn_bert_large_sampled_rows(bert_large_fp8):
    """Full BERT-large shape in the benchmark's launch configuration: the forward pass and the input
    gradient are row-wise independent given the weights, so the oracle chain is evaluated for a
    sample of token rows."""
    shape, blk, (X, W1, W2, G) = bert_large_fp8
    T, d, f = shape.tokens, shape.d_model, shape.d_ff
    rng = np.random.default_rng(1)
    rows = np.unique(np.concatenate([[0, 127, 128, T - 1], rng.integers(0, T, 28)]))
    sc = O.FFNScales.unconstrained(T, d, f)
    r = O.ffn_block(X[rows], W1, W2, G[rows], sc, operand="fp8")
    _compare_chain(blk, r, None, "fp8", rows=rows, weights=False)
    # statistics at initialisation (section "Unit Scaling": unit variance of activations and gradients)
    assert abs(blk.H.float().std().item() - 1) < 0.02
    assert abs(blk.Aq.float().std().item() - 1) < 0.03
    assert 0.9 < blk.dW1.std().item() < 1.2 and 0.9 < blk.dW2.std().item() < 1.2


def test_ffn_bert_large_full_oracle_chain(bert_large_fp8):
    """The same run against the full oracle chain (fp64 matmuls over all 8192 tokens), weight gradients included."""
    shape, blk, (X, W1, W2, G) = bert_large_fp8
    T, d, f = shape.tokens, shape.d_model, shape.d_ff
    sc = O.FFNScales.unconstrained(T, d, f)
    r = O.ffn_block(X, W1, W2, G, sc, operand="fp8")
    _compare_chain(blk, r, None, "fp8")


def test_ffn_bert_large_step_without_the_kept_pre_activation(bert_large_fp8):
    """The benchmark's configuration: the hidden-layer launch keeps the pre-activation on the SM and writes no copy
    (keep_h = False).  Every stored tensor must equal, bit for bit, the run above that also wrote the copy and
    was compared with the oracle; the H buffer stays untouched."""
    ffn, L, synth = _mods()
    shape, ref, tensors = bert_large_fp8
    blk = ffn.UnitScaledFFN(shape.tokens, shape.d_model, shape.d_ff)
    assert blk.fused_hidden and not blk.keep_h and blk.launches_per_step == 3
    blk.H.fill_(-7.0)
    blk.step(*[torch.from_numpy(t).cuda() for t in tensors])
    blk.check()
    for name in ("Xq", "W1q", "W2q", "Gq", "Aq", "dHq", "R", "dX", "dW1", "dW2"):
        a, b = getattr(blk, name), getattr(ref, name)
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), name
    assert bool((blk.H == -7.0).all())


@pytest.mark.parametrize("sigma", [2.0 ** 8, 2.0 ** -8])
def test_ffn_saturation_and_underflow_in_fused_cast(sigma):
    """X ~ N(0, sigma^2): sigma = 2^8 saturates part of q_E4(X) and of the fused A cast; sigma = 2^-8
    pushes X into E4M3's subnormal range.  Codes must still agree with the oracle's."""
    ffn, L, synth = _mods()
    shape = synth.FFN_SMALL
    blk, tensors = _run(shape, "fp8", seed=3, sigma_x=sigma)
    r = _oracle(shape, tensors, "fp8")
    want = F.quantise_codes(tensors[0], F.E4M3)
    assert np.array_equal(U.codes_of(blk.Xq), want)
    if sigma > 1:
        assert ((want & 0x7F) == 0x7E).mean() > 0.02           # some inputs clip to +-448
        assert ((r.Aq_codes & 0x7F) == 0x7E).mean() > 0.01     # and the fused GELU output saturates too
    else:
        assert ((want & 0x78) == 0).mean() > 0.5               # mostly subnormal / zero codes
    dA = U.code_deltas(blk.Aq, r.Aq_codes, "e4m3")
    tol = TOL * max(1.0, np.abs(r.dW2).max()) + blk.sc.beta_w * U.propagated(dA.T, r.Gq, "a")
    U.assert_close_stored(blk.dW2, r.dW2, "f32", tol, "dW2")


def test_step_on_three_streams_equals_step_on_one_stream():
    """The multi-stream issue order changes when kernels run, not what they compute: bit-identical outputs,
    eagerly and from a captured graph."""
    ffn, L, synth = _mods()
    shape = synth.FFN_RAGGED
    tensors = [torch.from_numpy(t).cuda() for t in synth.ffn_tensors(shape, seed=5)]
    outs = []
    for concurrent in (False, True):
        blk = ffn.UnitScaledFFN(shape.tokens, shape.d_model, shape.d_ff)
        blk.concurrent = concurrent
        blk.step(*tensors)
        blk.check()
        eager = [t.clone() for t in (blk.R, blk.dX, blk.dW1, blk.dW2)]
        g = blk.capture(*tensors)
        for t in (blk.R, blk.dX, blk.dW1, blk.dW2):
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        blk.check()
        for a, b in zip(eager, (blk.R, blk.dX, blk.dW1, blk.dW2)):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
        outs.append(eager)
    for a, b in zip(*outs):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("operand", ["fp8", "bf16", "fp16"])
def test_one_block_stepped_with_other_tensors_equals_new_blocks(operand):
    """The prepared calls of a block take whatever tensors each pass is given: other addresses, types and (16-bit operands)
    row pitches, against the single launches of a block of its own."""
    from paper_2303_11257_b200 import ffn
    T, d, f = 272, 144, 336
    block = ffn.UnitScaledFFN(T, d, f, operand=operand)
    for seed, dtype, pad in ((0, torch.float32, 0), (1, torch.bfloat16, 0), (2, torch.float32, 16 if operand != "fp8" else 0)):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = [torch.randn((r, c + pad), generator=g, device="cuda").to(dtype)[:, :c] for r, c in ((T, d), (d, f), (f, d), (T, d))]
        block.step(*x)
        other = ffn.UnitScaledFFN(T, d, f, operand=operand)
        other.grouped = other.fused_casts = False
        other.step(*x)
        block.check()
        other.check()
        for a, b in zip((block.R, block.dX, block.dW1, block.dW2), (other.R, other.dX, other.dW1, other.dW2)):
            assert torch.equal(a, b)
        block.forward(x[0])                                    # evaluation with the weights of that step
        assert torch.equal(block.R, other.R)
