"""The prepared calls of a block (lib.Plan): laid out once, their input slots refilled on every pass, laid out again when
a buffer or a value they were made for changes.  No GPU: the calls are inspected, not issued."""
import copy
import gc
import weakref

import pytest
import torch

from paper_2303_11257_b200 import encoder, ffn
from paper_2303_11257_b200 import lib as L


def test_slots_follow_the_inputs_and_calls_are_laid_out_once():
    own = (torch.zeros(4, 8), torch.zeros(4, 8))
    p = L.Plan(own, (1.0,))
    made = []

    def lay_out(plan):
        made.append(1)
        yield plan.cast_multi(["X", own[0]], own)
        yield L.Call("us_cast_fp8", plan.slot("X"), 1.0, L.mat(own[1]))

    for x in (torch.zeros(4, 8), torch.zeros(4, 16)[:, :8], torch.zeros(2, 3, dtype=torch.bfloat16)):
        p.put("X", x)
        calls = list(p.calls(lay_out))
        src, m = calls[0].keep[1], calls[1].keep[0]
        for got in (src[0], m):
            assert (got.ptr, got.dtype, got.rows, got.cols, got.ld) == L.describe(x)
        assert src[1].ptr == own[0].data_ptr()
    assert len(made) == 1
    assert p.same(own, (1.0,)) and not p.same(own, (2.0,))
    assert not p.same((own[0], own[1].clone()), (1.0,))


def test_a_pass_that_ends_early_is_laid_out_again_and_a_plan_keeps_nothing_but_its_buffers():
    own = (torch.zeros(2, 16),)

    class Block:
        def lay_out(self, plan):
            yield L.Call("us_cast_fp8", plan.slot("X"), 1.0, L.mat(own[0]))
            yield L.Call("us_cast_fp8", plan.slot("X"), 1.0, L.mat(own[0]))

    b = Block()
    b.plan = L.Plan(own, ())
    b.plan.put("X", own[0])
    next(iter(b.plan.calls(b.lay_out)))
    assert b.plan.done is None
    assert len(list(b.plan.calls(b.lay_out))) == 2 and len(b.plan.slots["X"]) == 2
    gone = weakref.ref(b)
    gc.disable()
    try:
        del b
        assert gone() is None
    finally:
        gc.enable()


class _Recorder:
    """Stands in for the library: notes every call (name, arguments) and returns a status for it."""

    def __init__(self, status=lambda name, args: L.US_OK):
        self.calls, self.status = [], status

    def __getattr__(self, name):
        def call(*args):
            self.calls.append((name, args))
            return self.status(name, args)
        return call

    def names(self):
        return [n for n, _ in self.calls]


def _ffn(**kw):
    return ffn.UnitScaledFFN(64, 32, 64, device="cpu", **kw), [torch.zeros(s) for s in ((64, 32), (32, 64), (64, 32), (64, 32))]


def _layer(**kw):
    kw = {"fused_attention": True, **kw}
    x = [torch.zeros(s) for s in ((128, 128), (128, 384), (128, 128), (128, 256), (256, 128), (128, 128))]
    return encoder.UnitScaledEncoderLayer(2, 64, 128, 2, 256, device="cpu", **kw), x


def _out_ptrs(rec):
    return {a._obj.ptr for _, args in rec.calls for a in args if isinstance(getattr(a, "_obj", None), L.us_mat)}


@pytest.mark.parametrize("make", [_ffn, _layer])
def test_blocks_are_copied_before_and_after_a_step(make, monkeypatch):
    """Prepared calls point into the object's buffers: they stay with it, and a copy lays out its own."""
    block, x = make()
    rec = _Recorder()
    for stepped in (False, True):
        if stepped:
            monkeypatch.setattr(L, "_lib", rec)
            block.step(*x, stream=0)
        other = copy.deepcopy(block)
        assert other.dX.data_ptr() != block.dX.data_ptr()
    first, rec.calls = _out_ptrs(rec), []
    other.step(*x, stream=0)
    mine = {t.data_ptr() for t in block._owned()}
    assert first & mine and not _out_ptrs(rec) & mine


GROUP, CAST = "us_linear_group_any", "us_cast_multi"


def _refuse(name, status):
    return lambda n, args: status if n == name else L.US_OK


@pytest.mark.parametrize("norm", [None, "post"])
def test_a_refused_group_goes_out_singly_and_nothing_is_issued_twice(norm, monkeypatch):
    """More tiles than the work list of the grouped launch holds: the calls of that step are the others, each once, and the
    group's GEMMs in its place -- in the first step and in later ones."""
    ln = [torch.ones(128)] * 4 if norm else None
    (layer, x), (other, _) = _layer(norm=norm), _layer(norm=norm)
    rec = _Recorder()
    monkeypatch.setattr(L, "_lib", rec)
    layer.step(*x, stream=0, ln=ln)
    want = []
    for name, args in rec.calls:
        want.append(name)
        if name == GROUP:
            want += [("us_linear_fwd", "us_linear_bwd_x", "us_linear_bwd_w")[c.op] for c in args[1]]
    refusing = _Recorder(_refuse(GROUP, L.US_ERR_UNSUPPORTED))
    monkeypatch.setattr(L, "_lib", refusing)
    for _ in range(2):
        other.step(*x, stream=0, ln=ln)
        assert refusing.names() == want
        refusing.calls.clear()


def test_a_block_whose_group_is_refused_finishes_the_step_and_takes_the_general_form_from_then_on(monkeypatch):
    block, x = _ffn()
    rec = _Recorder(_refuse(GROUP, L.US_ERR_UNSUPPORTED))
    monkeypatch.setattr(L, "_lib", rec)
    block.step(*x, stream=0)
    assert rec.names() == [CAST, "us_ffn_hidden_any", GROUP, "us_linear_bwd_w", "us_linear_bwd_w", "us_linear_fwd", "us_linear_bwd_x"]
    assert not block.grouped
    rec.calls.clear()
    block.step(*x, stream=0)
    assert GROUP not in rec.names() and rec.names().count("us_linear_bwd_w") == 2


def test_padded_inputs_of_a_16_bit_block_cost_one_refused_call_and_no_new_plan(monkeypatch):
    block, x = _ffn(operand="bf16")
    rec = _Recorder(_refuse(CAST, L.US_ERR_UNSUPPORTED))
    monkeypatch.setattr(L, "_lib", rec)
    block.step(*x, stream=0)
    plan = block._plans["step"]
    laid_out = plan.done
    rec.calls.clear()
    block.step(*x, stream=0)
    assert rec.names() == [CAST] + 4 * ["us_residual_add"] + ["us_ffn_hidden_any", GROUP]
    assert block._plans["step"] is plan and laid_out is not None and plan.done is laid_out


def test_what_the_cast_of_an_fp8_block_refuses_stays_refused(monkeypatch):
    for block, x in (_ffn(), _layer()):
        rec = _Recorder(_refuse(CAST, L.US_ERR_UNSUPPORTED))
        with monkeypatch.context() as m:
            m.setattr(L, "_lib", rec)
            with pytest.raises(L.UnitScaleError) as e:
                block.step(*x, stream=0)
        assert e.value.status == L.US_ERR_UNSUPPORTED and rec.names() == [CAST]


def test_the_first_pass_issues_its_first_call_before_it_makes_what_later_ones_need(monkeypatch):
    layer, x = _layer()
    rec, heads, early = _Recorder(), layer._heads, []
    monkeypatch.setattr(layer, "_heads", lambda *a: (early.append(len(rec.calls)), heads(*a))[1], raising=False)
    monkeypatch.setattr(L, "_lib", rec)
    layer.step(*x, stream=0)
    assert early and min(early) >= 2 and rec.names()[:2] == [CAST, "us_linear_fwd"]


@pytest.mark.parametrize("slen,fp8,yes,no", [
    (128, False, (1, 5000), ()), (144, False, (37, 80), (1, 36, 81)), (144, True, (37, 5000), (36,)), (192, False, (37, 80), (36, 81)), (208, False, (37, 5000), (36,)), (256, True, (37,), (36,)),
    (272, False, (), (8, 33, 256)), (336, False, (20, 33, 50, 66), (19, 36, 96)), (448, False, (20, 40, 66, 192), (34, 36, 256)),
    (480, False, (38, 256), (36, 68)), (512, False, (20, 66, 96, 256), (8, 36, 68)), (512, True, (20, 66, 96), (36, 128, 256)), (336, True, (33, 50), (49, 96))])
def test_when_the_attention_backward_pass_is_one_launch(slen, fp8, yes, no):
    assert all(encoder.backward_in_one_launch(p, slen, fp8) for p in yes)
    assert not any(encoder.backward_in_one_launch(p, slen, fp8) for p in no)
