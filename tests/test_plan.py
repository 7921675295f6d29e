"""The prepared calls of a block (lib.Plan): laid out once, their input slots refilled on every pass, laid out again when
a buffer or a value they were made for changes.  No GPU: the calls are inspected, not issued."""
import gc
import weakref

import torch

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
