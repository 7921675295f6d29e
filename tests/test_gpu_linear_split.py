"""Linear ops whose contraction is shared by the CTAs of a cluster (few output tiles, long K): two, four and eight CTAs on tiles of 128 x 64
and 128 x 128, two and four CTA pairs on 256 x 256 (test_every_form says which call takes which), with rows, columns and K blocks that do
not divide.  A part of the contraction is a
float32 sum like the whole, so the bounds are those of the unshared kernels."""
import numpy as np
import pytest
import torch

from oracle import ops as O
from tests import util as U
from tests.test_gpu_linear_narrow import PAD, TOL, _operands

pytestmark = pytest.mark.gpu

# rows, contraction, columns
SHAPES = [(1, 2576, 16), (48, 4096, 1024), (130, 5008, 700), (300, 5008, 690), (500, 6160, 1300), (2048, 6400, 1024), (1000, 8208, 700)]


@pytest.mark.parametrize("op,fmt,out_fmt", [("fwd", "e4m3", "bf16"), ("fwd", "bf16", "f32"), ("fwd", "fp16", "e4m3"), ("bwd_x", "e4m3", "f32"),
                                            ("bwd_x", "bf16", "bf16"), ("bwd_w", "e4m3", "f32"), ("bwd_w", "bf16", "f32")])
@pytest.mark.parametrize("rows,k,cols", SHAPES)
def test_shared_contraction(op, fmt, out_fmt, rows, k, cols):
    from paper_2303_11257_b200 import lib as L, synth
    fb = "e5m2" if fmt == "e4m3" and op != "fwd" else fmt
    A, B, val, scale = _operands(L, synth, op, rows, k, cols, 81, fmt, fb)
    ws, fn = L.new_workspace(), getattr(L, "us_linear_" + op)
    out, again = U.empty(rows, cols, out_fmt, PAD(cols)), U.empty(rows, cols, out_fmt, PAD(cols))
    tol = TOL * max(1.0, np.abs(val).max() / 4)
    fn(A, B, scale, out, ws)
    for _ in range(3):
        fn(A, B, scale, again, ws)
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(out, val, out_fmt, tol, f"{op} plain")
    assert torch.equal(out.contiguous().view(torch.uint8), again.contiguous().view(torch.uint8))
    if PAD(cols) > cols:
        assert not out.as_strided((rows, PAD(cols)), (PAD(cols), 1))[:, cols:].contiguous().view(torch.uint8).any()
    for skip_fmt in ("f32", "bf16"):
        sk = synth.normal(81, 2, (rows, cols))
        out = U.empty(rows, cols, out_fmt, PAD(cols))
        fn(A, B, scale, out, ws, L.epilogue(skip=U.to_device(sk, skip_fmt, PAD(cols)), skip_coef=0.8, out_coef=0.6))
        assert L.us_workspace_status(ws) == 0
        U.assert_close_stored(out, O.weighted_add(U.values_of(sk, skip_fmt), val, np.float32(0.8), np.float32(0.6)), out_fmt, tol, f"{op} residual {skip_fmt}")


@pytest.mark.parametrize("rows,k,cols", [(48, 4096, 1024), (2048, 6400, 1024)])
def test_shared_contraction_with_a_copy_in_fp8(rows, k, cols):
    from paper_2303_11257_b200 import lib as L, synth
    X, W, val, scale = _operands(L, synth, "fwd", rows, k, cols, 82, "e4m3", "e4m3")
    ws, out, q = L.new_workspace(), U.empty(rows, cols, "bf16"), U.empty(rows, cols, "e4m3")
    sk = synth.normal(82, 2, (rows, cols))
    plan = L.Plan((), ())
    ep = L.epilogue(skip=U.to_device(sk, "f32"), skip_coef=0.8, out_coef=0.6)
    L.Call("us_linear_fwd_cast", plan.mat(X), plan.mat(W), scale, ep, plan.mat(out), plan.mat(q), ws.data_ptr(), ws.numel())(L.current_stream())
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(out, O.weighted_add(U.values_of(sk, "f32"), val, np.float32(0.8), np.float32(0.6)), "bf16", TOL * max(1.0, np.abs(val).max() / 4), "residual")
    assert torch.equal(q.view(torch.uint8), out.float().clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8))


def test_waits_that_run_out_in_a_cluster():
    """Operand loads withheld: every CTA's waits run out, the cluster's barriers are passed all the same, the status says so, and
    the next call is correct."""
    from paper_2303_11257_b200 import lib as L, synth
    for rows, k, cols in ((48, 4096, 1024), (2048, 6400, 1024)):
        X, W, val, scale = _operands(L, synth, "fwd", rows, k, cols, 83, "e4m3", "e4m3")
        ws, out = L.new_workspace(), U.empty(rows, cols, "bf16")
        L.us_test_linear_fwd_starved(X, W, scale, out, ws, 2000)
        assert L.us_workspace_status(ws) == L.US_ERR_TIMEOUT
        ws.zero_()
        L.us_linear_fwd(X, W, scale, out, ws)
        assert L.us_workspace_status(ws) == 0
        U.assert_close_stored(out, val, "bf16", TOL * max(1.0, np.abs(val).max() / 4), "after")


# Every form: (columns of a tile, CTAs of a pair, shares) on 148 SMs, and a forward call that takes it.
FORMS = {(64, 1, 2): ("e4m3", 300, 5024, 690), (64, 1, 4): ("e4m3", 48, 4096, 1024), (64, 1, 8): ("bf16", 1, 2576, 16), (128, 1, 2): ("bf16", 500, 6160, 1300),
         (128, 1, 4): ("bf16", 300, 5008, 690), (128, 1, 8): ("e4m3", 128, 32768, 1280), (256, 2, 2): ("e4m3", 2048, 6400, 1024), (256, 2, 4): ("bf16", 1000, 8208, 700)}


@pytest.mark.parametrize("form", list(FORMS), ids=str)
def test_every_form(form):
    """The form is the one that is meant; its result; its waits when they run out in every CTA, and in one CTA only (of a pair the odd one):
    the cluster's barriers are passed all the same, the status says so, and the next call has the bits of the first."""
    from paper_2303_11257_b200 import lib as L, synth
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the choice depends on the number of SMs")
    fmt, rows, k, cols = FORMS[form]
    X, W, val, scale = _operands(L, synth, "fwd", rows, k, cols, 83, fmt, fmt)
    ws, out = L.new_workspace(), U.empty(rows, cols, "f32", PAD(cols))
    assert L.us_test_linear_tiling(L.US_OP_FWD, X, W, out, ws) == form
    L.us_linear_fwd(X, W, scale, out, ws)
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(out, val, "f32", TOL * max(1.0, np.abs(val).max() / 4), "first")
    first = out.clone()
    ctas = form[1] * form[2]
    for cta in (-1, 1, ctas - 1):
        L.us_test_linear_fwd_starved_cta(X, W, scale, out, ws, 2000, cta, 0)
        assert L.us_workspace_status(ws) == L.US_ERR_TIMEOUT, cta
        ws.zero_()
        L.us_linear_fwd(X, W, scale, out, ws)
        assert L.us_workspace_status(ws) == 0 and torch.equal(out, first), cta


@pytest.mark.parametrize("fmt,b,m,n", [("e4m3", 16000, 128, 400), ("bf16", 9008, 256, 768)])
def test_waits_that_run_out_in_the_shared_launch_of_a_group(fmt, b, m, n):
    from paper_2303_11257_b200 import lib as L, synth
    dev = lambda i, shape: U.to_device(synth.normal(95 + i, 0, shape), fmt, PAD(shape[1]))
    X, W, G, ws = dev(0, (b, m)), dev(1, (m, n)), dev(2, (b, n)), L.new_workspace()
    outs = [U.empty(m, n, "f32"), U.empty(m, n, "bf16", PAD(n)), U.empty(b, n, "bf16", PAD(n)), U.empty(b, m, "bf16")]
    calls = [L.linear_call(L.US_OP_BWD_W, X, G, b ** -0.5, outs[0]), L.linear_call(L.US_OP_BWD_W, X, G, b ** -0.5, outs[1]),
             L.linear_call(L.US_OP_FWD, X, W, 0.1, outs[2]), L.linear_call(L.US_OP_BWD_X, G, W, 0.1, outs[3])]
    assert L.us_linear_group_launches(calls) == 2
    L.us_linear_group_any(calls, ws)
    assert L.us_workspace_status(ws) == 0
    first = [t.clone() for t in outs]
    for cta in (-1, 1, 3):
        L.us_test_linear_group_starved(calls, ws, 2000, cta, 0)
        assert L.us_workspace_status(ws) == L.US_ERR_TIMEOUT, cta
        ws.zero_()
        L.us_linear_group_any(calls, ws)
        assert L.us_workspace_status(ws) == 0 and all(torch.equal(t.view(torch.uint8), f.view(torch.uint8)) for t, f in zip(outs, first)), cta


@pytest.mark.parametrize("fmt", ["e4m3", "bf16"])
@pytest.mark.parametrize("b,m,n", [(16000, 128, 400), (8200, 272, 144), (6500, 64, 80)])
def test_grouped_launch_whose_long_contractions_are_shared(fmt, b, m, n):
    """The weight gradients of many tokens beside the other two products of a step, with a residual and its copy in FP8: against the single
    entry points, whose sums are float32 sums in another order (2e-6 of the largest result, one step of the stored format)."""
    from paper_2303_11257_b200 import lib as L, synth
    ws = L.new_workspace()
    dev = lambda i, shape: U.to_device(synth.normal(90 + i, 0, shape), fmt, PAD(shape[1]))
    X, W, G, skip = dev(0, (b, m)), dev(1, (m, n)), dev(2, (b, n)), U.to_device(synth.normal(93, 0, (b, m)), "f32")
    ep = lambda: L.epilogue(skip=skip, skip_coef=0.8, out_coef=0.6)
    s = b ** -0.5
    outs = [[U.empty(m, n, "f32"), U.empty(b, n, "bf16", PAD(n)), U.empty(b, m, "bf16"), U.empty(m, n, "fp16", PAD(n))] for _ in range(3)]
    q = U.empty(b, m, "e5m2")
    for o in outs[:2]:
        plan = L.Plan((), ())
        plan.group([(L.US_OP_BWD_W, X, G, s, o[0], None, None), (L.US_OP_FWD, X, W, 0.1, o[1], None, None),
                    (L.US_OP_BWD_X, G, W, 0.1, o[2], skip, (0.8, 0.6)), (L.US_OP_BWD_W, X, G, s, o[3], None, None)], ws, {2: q})(L.current_stream())
    o = outs[2]
    L.us_linear_bwd_w(X, G, s, o[0], ws)
    L.us_linear_fwd(X, W, 0.1, o[1], ws)
    L.us_linear_bwd_x(G, W, 0.1, o[2], ws, ep())
    L.us_linear_bwd_w(X, G, s, o[3], ws)
    assert L.us_workspace_status(ws) == 0
    for a, r in zip(outs[0], outs[1]):
        assert torch.equal(a.contiguous().view(torch.uint8), r.contiguous().view(torch.uint8))
    ref = U.host_values(o[0])
    assert np.abs(U.host_values(outs[0][0]) - ref).max() <= 2e-6 * np.abs(ref).max()
    U.assert_close_stored(outs[0][3], ref, "fp16", 2e-6 * np.abs(ref).max(), "fp16 weight gradient")
    for i in (1, 2):
        assert torch.equal(outs[0][i].contiguous().view(torch.uint8), o[i].contiguous().view(torch.uint8))
    assert torch.equal(q.view(torch.uint8), outs[0][2].float().clamp(-57344, 57344).to(torch.float8_e5m2).view(torch.uint8))


def test_grouped_launch_leaves_longer_contractions_than_were_measured_alone():
    """Beyond 8192 K blocks a contraction is not shared, nor is one beside it: the bits are those of the single entry point, one accumulator
    per tile."""
    from paper_2303_11257_b200 import lib as L
    ws = L.new_workspace()
    torch.manual_seed(84)
    long, short = (8192 + 40) * 128, 120 * 128
    A, B = ((torch.randn(long, 16, device="cuda")).to(torch.float8_e4m3fn) for _ in range(2))
    one, two, alone = (torch.empty(16, 16, device="cuda") for _ in range(3))
    L.us_linear_group_any([L.linear_call(L.US_OP_BWD_W, A, B, long ** -0.5, one), L.linear_call(L.US_OP_BWD_W, A[:short], B[:short], short ** -0.5, two)], ws)
    L.us_linear_bwd_w(A, B, long ** -0.5, alone, ws)
    assert L.us_workspace_status(ws) == 0
    assert torch.equal(one, alone)
    assert (two - (A[:short].float().T @ B[:short].float()) * short ** -0.5).abs().max() <= 1e-3
