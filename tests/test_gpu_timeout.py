"""The bounded-wait failure path of the linear kernels, driven without faulting the GPU.

us_test_linear_fwd_starved launches the forward kernel with its operand loads withheld and a short
wait limit: nothing is in flight, every role's wait runs out, the kernel raises the status word, frees its
tensor memory and returns.  The context must stay usable: after clearing the word, an ordinary call
on the same workspace has to match the oracle."""
import time

import numpy as np
import pytest
import torch

from oracle import ops as O
from oracle import scales as S
from tests import util as U

pytestmark = pytest.mark.gpu
TOL = 2e-3
US_ERR_TIMEOUT = 6


@pytest.mark.parametrize("shape", [(96, 64, 80), (520, 272, 1040)])      # one 128-row tile; CTA-pair tiles (256 x 256)
def test_starved_launch_times_out_and_the_next_call_is_correct(shape):
    from paper_2303_11257_b200 import lib as L, synth
    b, m, n = shape
    X, W, _ = synth.linear_tensors(b, m, n, 31)
    Xt, Wt = U.to_device(X, "e4m3"), U.to_device(W, "e4m3")
    alpha, _, _ = S.linear_scales(b, m, n)
    ws = L.new_workspace()
    junk = U.empty(b, n, "f32")
    L.us_test_linear_fwd_starved(Xt, Wt, float(alpha), junk, ws, wait_limit=2000)
    assert L.us_workspace_status(ws) == US_ERR_TIMEOUT            # synchronises: the kernel has returned by itself
    # the word is sticky until the caller clears it
    out = U.empty(b, n, "f32")
    L.us_linear_fwd(Xt, Wt, float(alpha), out, ws)
    assert L.us_workspace_status(ws) == US_ERR_TIMEOUT
    ref = O.linear_fwd(U.values_of(X, "e4m3"), U.values_of(W, "e4m3"), alpha)
    U.assert_close_stored(out, ref, "f32", TOL, "call after a timed-out launch")   # the kernel itself ran normally
    ws.zero_()
    out2 = U.empty(b, n, "bf16")
    L.us_linear_fwd(Xt, Wt, float(alpha), out2, ws)
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(out2, ref, "bf16", TOL, "call after clearing the word")
    # tensor memory was released: a kernel that needs all of it (two 256-column accumulators per SM) still runs
    big = U.empty(512, 512, "f32")
    Xb, Wb, _ = synth.linear_tensors(512, 256, 512, 32)
    L.us_linear_fwd(U.to_device(Xb, "e4m3"), U.to_device(Wb, "e4m3"), 1.0 / 16, big, ws)
    assert L.us_workspace_status(ws) == 0
    refb = O.linear_fwd(U.values_of(Xb, "e4m3"), U.values_of(Wb, "e4m3"), 1.0 / 16)
    U.assert_close_stored(big, refb, "f32", TOL, "full-width kernel after the timed-out launch")


def test_starved_launch_argument_checks():
    from paper_2303_11257_b200 import lib as L
    ws = L.new_workspace()
    X, W, Y = U.empty(32, 64, "e4m3"), U.empty(64, 48, "e4m3"), U.empty(32, 48, "f32")
    for bad in (0, 1 << 17):
        with pytest.raises(L.UnitScaleError) as e:
            L.us_test_linear_fwd_starved(X, W, 1.0, Y, ws, wait_limit=bad)
        assert e.value.status == 1
    assert L.us_workspace_status(ws) == 0


def _bytes(*ts):
    return [t.contiguous().view(torch.uint8).clone() for t in ts]


def _starve_and_repeat(L, ws, starve, run, outs):
    """The results of a call before and after launches that starved are the same bits, and each of those is reported."""
    run()
    want = _bytes(*outs)
    for cta, tiles in ((-1, 1), (-1, 2), (1, 0), (1, 1), (1, 2)):
        starve(cta, tiles)
        assert L.us_workspace_status(ws) == US_ERR_TIMEOUT, (cta, tiles)
        ws.zero_()
        for t in outs:
            t.view(torch.uint8).zero_()
        run()
        assert L.us_workspace_status(ws) == 0, (cta, tiles)
        assert all(torch.equal(a, b) for a, b in zip(_bytes(*outs), want)), (cta, tiles)


@pytest.mark.parametrize("out_fmt", ["e4m3", "bf16", "f32"])
def test_pairs_whose_operands_stop_after_some_tiles(out_fmt):
    """240 tiles of 256 x 256, three or four per CTA pair: a pair gives up with accumulators handed back that nobody takes any more, or
    because only its odd CTA gets no operands; both CTAs leave in order and the next call is correct."""
    from paper_2303_11257_b200 import lib as L, synth
    X, W, _ = synth.linear_tensors(3840, 144, 4096, 33)
    X, W, ws, out = U.to_device(X, "e4m3"), U.to_device(W, "e4m3"), L.new_workspace(), U.empty(3840, 4096, out_fmt)
    _starve_and_repeat(L, ws, lambda cta, tiles: L.us_test_linear_fwd_starved_cta(X, W, 1 / 12, out, ws, 2000, cta, tiles),
                       lambda: L.us_linear_fwd(X, W, 1 / 12, out, ws), [out])


def test_hidden_pairs_whose_operands_stop_after_some_tiles():
    from paper_2303_11257_b200 import lib as L, synth
    d = lambda i, shape, fmt: U.to_device(synth.normal(34, i, shape), fmt)
    X, W1, G, W2 = d(0, (3840, 144), "e4m3"), d(1, (144, 4096), "e4m3"), d(2, (3840, 144), "e5m2"), d(3, (4096, 144), "e4m3")
    ws, A, dH = L.new_workspace(), U.empty(3840, 4096, "e4m3"), U.empty(3840, 4096, "e5m2")
    _starve_and_repeat(L, ws, lambda cta, tiles: L.us_test_ffn_hidden_starved_cta(X, W1, G, W2, A, dH, ws, 2000, cta, tiles),
                       lambda: L.us_ffn_hidden(X, W1, 1 / 12, G, W2, 1 / 12, 1.0, 1.7, 1.5, A, dH, ws), [A, dH])


@pytest.mark.parametrize("fmt", ["e4m3", "bf16"])
def test_grouped_pairs_whose_operands_stop_after_some_tiles(fmt):
    from paper_2303_11257_b200 import lib as L, synth
    d = lambda i, shape: U.to_device(synth.normal(35, i, shape), fmt)
    X, W, G, skip = d(0, (3840, 144)), d(1, (144, 4096)), d(2, (3840, 4096)), U.to_device(synth.normal(35, 3, (3840, 144)), "f32")
    ws, Y, dX = L.new_workspace(), U.empty(3840, 4096, "bf16"), U.empty(3840, 144, "bf16")
    calls = [L.linear_call(L.US_OP_FWD, X, W, 1 / 12, Y), L.linear_call(L.US_OP_BWD_X, G, W, 1 / 64, dX, L.epilogue(skip=skip, skip_coef=0.8, out_coef=0.6))]
    _starve_and_repeat(L, ws, lambda cta, tiles: L.us_test_linear_group_starved(calls, ws, 2000, cta, tiles),
                       lambda: L.us_linear_group_any(calls, ws), [Y, dX])


def test_partly_starved_launch_argument_checks():
    from paper_2303_11257_b200 import lib as L
    ws = L.new_workspace()
    X, W, Y = U.empty(32, 64, "e4m3"), U.empty(64, 48, "e4m3"), U.empty(32, 48, "f32")
    for limit, cta, tiles in ((0, -1, 0), (1 << 17, -1, 0), (100, -2, 0), (100, 8, 0), (100, 0, -1), (100, 0, 1025)):
        with pytest.raises(L.UnitScaleError) as e:
            L.us_test_linear_fwd_starved_cta(X, W, 1.0, Y, ws, limit, cta, tiles)
        assert e.value.status == 1
    assert L.us_workspace_status(ws) == 0


def _starve_linear(L, ws):
    X, W, Y = U.empty(96, 64, "e4m3"), U.empty(64, 80, "e4m3"), U.empty(96, 80, "f32")
    return lambda: L.us_test_linear_fwd_starved(X, W, 1.0, Y, ws, wait_limit=500)


def _starve_hidden(L, ws):
    X, W1, A = U.empty(200, 144, "e4m3"), U.empty(144, 336, "e4m3"), U.empty(200, 336, "e4m3")
    G, W2, dH = U.empty(200, 144, "e5m2"), U.empty(336, 144, "e4m3"), U.empty(200, 336, "e5m2")
    return lambda: L.us_test_ffn_hidden_starved(X, W1, G, W2, A, dH, ws, wait_limit=500)


@pytest.mark.parametrize("make", [_starve_linear, _starve_hidden])
def test_the_time_of_the_previous_kernel_is_not_counted_against_a_bounded_wait(make):
    """A launch that overlaps a long predecessor (one tile, a contraction of 2^22) must begin to count its polls when that
    has finished: half way through the predecessor its status word is still clear, although its limit is far shorter."""
    from paper_2303_11257_b200 import lib as L
    k = 1 << 22
    X, W, Y = U.empty(16, k, "e4m3"), U.empty(k, 16, "e4m3"), U.empty(16, 16, "f32")
    ws_long, ws, seen = L.new_workspace(), L.new_workspace(), torch.full((256,), 255, dtype=torch.uint8).pin_memory()
    other, starve = torch.cuda.Stream(), make(L, ws)
    L.us_linear_fwd(X, W, 1.0, Y, ws_long)
    starve()                                              # kernels loaded, allocations made
    torch.cuda.synchronize()
    ws.zero_()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    L.us_linear_fwd(X, W, 1.0, Y, ws_long)
    torch.cuda.synchronize()
    alone = time.perf_counter() - t0
    assert alone > 2e-3                                        # far longer than 500 polls
    L.us_linear_fwd(X, W, 1.0, Y, ws_long)
    starve()
    time.sleep(alone / 2)
    with torch.cuda.stream(other):
        seen.copy_(ws.view(torch.uint8)[:256], non_blocking=True)
    other.synchronize()
    assert not seen.any()
    assert L.us_workspace_status(ws) == US_ERR_TIMEOUT and L.us_workspace_status(ws_long) == 0
