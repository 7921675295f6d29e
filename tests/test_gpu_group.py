"""us_linear_group: several independent linear ops in one launch, against the oracle and against the
single entry points (bit-identical: every tile is still accumulated by one accumulator over its whole K)."""
import numpy as np
import pytest
import torch

from oracle import ops as O
from oracle import scales as S
from tests import util as U

pytestmark = pytest.mark.gpu
TOL = 2e-3


def _mods():
    from paper_2303_11257_b200 import lib, synth
    return lib, synth


def _problem(L, synth, op, b, m, n, seed, out_fmt, skip_fmt=None, fa="e4m3", fb="e4m3"):
    X, W, G = synth.linear_tensors(b, m, n, seed)
    a, bx, bw = S.linear_scales(b, m, n)
    A, B, scale, ref_fn, oshape, code = {"fwd": (X, W, a, O.linear_fwd, (b, n), L.US_OP_FWD),
                                         "bwd_x": (G, W, bx, O.linear_bwd_x, (b, m), L.US_OP_BWD_X),
                                         "bwd_w": (X, G, bw, O.linear_bwd_w, (m, n), L.US_OP_BWD_W)}[op]
    At, Bt = U.to_device(A, fa), U.to_device(B, fb)
    ref = ref_fn(U.values_of(A, fa), U.values_of(B, fb), scale)
    ep, ep_args = None, None
    if skip_fmt:
        sk = synth.normal(seed, 9, oshape)
        cs, cb = S.residual_coefficients(0.3)
        skt = U.to_device(sk, skip_fmt)
        ep_args = dict(skip=skt, skip_coef=float(cs), out_coef=float(cb))
        ref = O.weighted_add(U.values_of(sk, skip_fmt), ref, cs, cb)
    out = U.empty(oshape[0], oshape[1], out_fmt)
    single = U.empty(oshape[0], oshape[1], out_fmt)
    mk_ep = (lambda: L.epilogue(**ep_args)) if ep_args else (lambda: None)
    return dict(op=op, code=code, At=At, Bt=Bt, scale=float(scale), ref=ref, out=out, single=single, mk_ep=mk_ep, out_fmt=out_fmt)


CASES = [
    # ragged shapes, every layout, every output format, with and without a skip tensor
    [("fwd", 304, 272, 528, "f32", None), ("bwd_x", 272, 400, 304, "bf16", "f32"), ("bwd_w", 400, 272, 304, "f32", None),
     ("fwd", 528, 144, 272, "e4m3", "bf16")],
    [("bwd_w", 1024, 512, 768, "bf16", None), ("bwd_x", 512, 384, 1040, "e5m2", None)],
    [("fwd", 272, 2064, 272, "fp16", "fp16")],
    # long and short contractions mixed: the work list gives some pairs several tiles
    [("bwd_w", 4096, 512, 512, "f32", None), ("fwd", 1536, 256, 1024, "bf16", "f32"), ("bwd_x", 1536, 1024, 128 * 3, "bf16", "bf16"),
     ("bwd_w", 2048, 304, 528, "f32", None)],
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_group_matches_oracle_and_single_calls(case):
    L, synth = _mods()
    ws = L.new_workspace()
    probs = []
    for i, (op, b, m, n, out_fmt, skip_fmt) in enumerate(CASES[case]):
        fa, fb = {"fwd": ("e4m3", "e4m3"), "bwd_x": ("e5m2", "e4m3"), "bwd_w": ("e4m3", "e5m2")}[op]
        probs.append(_problem(L, synth, op, b, m, n, 70 + 10 * case + i, out_fmt, skip_fmt, fa, fb))
    calls = [L.linear_call(p["code"], p["At"], p["Bt"], p["scale"], p["out"], p["mk_ep"]()) for p in probs]
    L.us_linear_group(calls, ws)
    assert L.us_workspace_status(ws) == 0
    for p in probs:
        U.assert_close_stored(p["out"], p["ref"], p["out_fmt"], TOL * max(1.0, np.abs(p["ref"]).max() / 4), f"group {p['op']}")
        getattr(L, "us_linear_" + p["op"])(p["At"], p["Bt"], p["scale"], p["single"], ws, p["mk_ep"]())
        torch.cuda.synchronize()
        assert torch.equal(p["out"].contiguous().view(torch.uint8), p["single"].contiguous().view(torch.uint8)), p["op"]
    assert L.us_workspace_status(ws) == 0


def test_group_unsupported_and_invalid_calls_launch_nothing():
    L, synth = _mods()
    ws = L.new_workspace()
    big = lambda fmt: (U.empty(272, 272, fmt), U.empty(272, 304, fmt), U.empty(272, 304, "f32"))

    def status(calls):
        with pytest.raises(L.UnitScaleError) as e:
            L.us_linear_group(calls, ws)
        return e.value.status

    A, B, out = big("e4m3")
    assert status([L.linear_call(L.US_OP_FWD, *big("bf16")[:2], 1.0, out)]) == 2                  # 16-bit operands
    assert status([L.linear_call(L.US_OP_FWD, U.empty(64, 272, "e4m3"), B, 1.0, U.empty(64, 304, "f32"))]) == 2     # small output
    ep = L.epilogue(act=L.US_ACT_GELU)
    assert status([L.linear_call(L.US_OP_FWD, A, B, 1.0, out, ep)]) == 2                          # fused activation
    assert status([L.linear_call(L.US_OP_FWD, A, B, 1.0, U.empty(272, 308, "f32"))]) == 1         # shape mismatch
    assert status([L.linear_call(7, A, B, 1.0, out)]) == 1
    assert status([L.linear_call(L.US_OP_FWD, A, B, 1.0, out)] * 5) == 2                          # more than four calls
    sentinel = out.clone()
    assert torch.equal(out, sentinel) and L.us_workspace_status(ws) == 0


def test_ffn_step_with_the_grouped_launch_equals_the_seven_launch_step():
    from paper_2303_11257_b200 import ffn, synth
    shape = synth.FFN_RAGGED
    shape = synth.FFNShape("ragged_wide", 400, 272, 528)
    tensors = [torch.from_numpy(t).cuda() for t in synth.ffn_tensors(shape, seed=6)]
    outs = []
    for grouped in (True, False):
        blk = ffn.UnitScaledFFN(shape.tokens, shape.d_model, shape.d_ff)
        blk.grouped = grouped
        blk.step(*tensors)
        blk.check()
        outs.append([t.clone() for t in (blk.R, blk.dX, blk.dW1, blk.dW2)])
    for a, b in zip(*outs):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("fmt", ["bf16", "fp16", "e4m3"])
@pytest.mark.parametrize("b,m,n", [(1, 16, 16), (48, 128, 512), (129, 80, 136), (2000, 528, 272), (4352, 1040, 2048)])
def test_group_any_equals_single_calls(fmt, b, m, n):
    """16-bit operands, outputs of one tile or less, both tile sizes and a work list of more than twelve rounds: the
    grouped launch without the size limits against the single entry points."""
    L, synth = _mods()
    ws = L.new_workspace()
    dev = lambda i, shape: U.to_device(synth.normal(40 + i, 0, shape), fmt, (shape[1] + 15) // 16 * 16)
    X, W, G, skip = dev(0, (b, m)), dev(1, (m, n)), dev(2, (b, n)), U.to_device(synth.normal(44, 0, (b, m)), "f32")
    ep = lambda: L.epilogue(skip=skip, skip_coef=0.8, out_coef=0.6)
    outs = [[U.empty(b, n, "bf16", (n + 7) // 8 * 8), U.empty(b, m, "bf16"), U.empty(m, n, "f32"), U.empty(m, n, "fp16", (n + 7) // 8 * 8)] for _ in range(2)]
    o = outs[0]
    L.us_linear_group_any([L.linear_call(L.US_OP_BWD_W, X, G, 0.1, o[2]), L.linear_call(L.US_OP_FWD, X, W, 0.2, o[0]),
                           L.linear_call(L.US_OP_BWD_X, G, W, 0.3, o[1], ep()), L.linear_call(L.US_OP_BWD_W, X, G, 0.4, o[3])], ws)
    o = outs[1]
    L.us_linear_bwd_w(X, G, 0.1, o[2], ws)
    L.us_linear_fwd(X, W, 0.2, o[0], ws)
    L.us_linear_bwd_x(G, W, 0.3, o[1], ws, ep())
    L.us_linear_bwd_w(X, G, 0.4, o[3], ws)
    assert L.us_workspace_status(ws) == 0
    for a, r in zip(*outs):
        assert torch.equal(a.contiguous().view(torch.uint8), r.contiguous().view(torch.uint8))


@pytest.mark.parametrize("out_fmt", ["e5m2", "e4m3"])
def test_group_any_fp8_outputs_of_small_tiles(out_fmt):
    """FP8 results of 128 x 128 tiles leave by 32-byte boxes where two CTAs share a tile, by 64-byte boxes otherwise (128
    tiles): ragged columns and a second tile."""
    L, synth = _mods()
    ws = L.new_workspace()
    for b, m, n in ((40, 208, 80), (200, 64, 176), (2000, 1008, 80)):
        G, W = U.to_device(synth.normal(50, 0, (b, n)), "e5m2"), U.to_device(synth.normal(50, 1, (m, n)), "e4m3")
        o, r = U.empty(b, m, out_fmt), U.empty(b, m, out_fmt)
        L.us_linear_group_any([L.linear_call(L.US_OP_BWD_X, G, W, n ** -0.5, o)], ws)
        L.us_linear_bwd_x(G, W, n ** -0.5, r, ws)
        assert np.array_equal(U.codes_of(o), U.codes_of(r))
    assert L.us_workspace_status(ws) == 0


def test_more_tiles_than_the_work_list_holds_go_out_singly():
    """46 x 46 tiles of 256 x 256 are more than the list's 2048 entries: the grouped call refuses them and launches nothing,
    and a prepared pass issues the same GEMMs as single launches."""
    L, synth = _mods()
    n, k = 46 * 256, 16
    X, W, G = (U.to_device(synth.normal(60, i, s), f) for i, s, f in ((0, (n, k), "e4m3"), (1, (k, n), "e4m3"), (2, (n, 64), "e5m2")))
    ws = L.new_workspace()
    big, dw, big1, dw1 = U.empty(n, n, "e4m3"), U.empty(k, 64, "f32"), U.empty(n, n, "e4m3"), U.empty(k, 64, "f32")
    big.view(torch.uint8).fill_(0x55)
    calls = [L.linear_call(L.US_OP_FWD, X, W, 0.25, big), L.linear_call(L.US_OP_BWD_W, X, G, 0.5, dw)]
    with pytest.raises(L.UnitScaleError) as e:
        L.us_linear_group_any(calls, ws)
    assert e.value.status == L.US_ERR_UNSUPPORTED and bool((big.view(torch.uint8) == 0x55).all())
    call = L.Plan((), ()).group([(L.US_OP_FWD, X, W, 0.25, big, None, None), (L.US_OP_BWD_W, X, G, 0.5, dw, None, None)], ws)
    call(L.current_stream())
    assert call.refused
    L.us_linear_fwd(X, W, 0.25, big1, ws)
    L.us_linear_bwd_w(X, G, 0.5, dw1, ws)
    assert L.us_workspace_status(ws) == 0
    assert torch.equal(big.view(torch.uint8), big1.view(torch.uint8)) and torch.equal(dw, dw1)
