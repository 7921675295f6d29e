"""Linear ops whose outputs are few tiles of 128 x 128: tiles of 128 x 64, and with at most 128 rows only as many rows of A in a
stage as there are (K-major A).  Every operand layout and width, every output format, every epilogue, at row counts around the eight-row
steps of A and column counts around the 64 of a tile and the 32 of a warp."""
import numpy as np
import pytest
import torch

from oracle import ops as O
from oracle import scales as S
from tests import util as U

pytestmark = pytest.mark.gpu
TOL = 2e-3
PAD = lambda c: (c + 15) // 16 * 16


def _operands(L, synth, op, rows, k, cols, seed, fa, fb):
    """A and B of the call whose output is rows x cols, the oracle's values of scale * A B and the scale."""
    sa, sb = {"fwd": ((rows, k), (k, cols)), "bwd_x": ((rows, k), (cols, k)), "bwd_w": ((k, rows), (k, cols))}[op]
    A, B = synth.normal(seed, 0, sa), synth.normal(seed, 1, sb)
    av, bv, scale = U.values_of(A, fa), U.values_of(B, fb), k ** -0.5
    ref = {"fwd": lambda: av @ bv, "bwd_x": lambda: av @ bv.T, "bwd_w": lambda: av.T @ bv}[op]()
    return U.to_device(A, fa, PAD(sa[1])), U.to_device(B, fb, PAD(sb[1])), scale * ref, scale


# rows, contraction, columns; the last two: more contraction than any ring of stages holds, and the most tiles (147 of 148 SMs)
SHAPES = [(1, 16, 16), (7, 80, 31), (8, 200, 33), (9, 128, 63), (48, 1024, 64), (65, 272, 65), (127, 400, 96), (128, 144, 97), (129, 304, 128),
          (300, 96, 200), (40, 6000, 80), (890, 272, 1300)]


@pytest.mark.parametrize("op", ["fwd", "bwd_x", "bwd_w"])
@pytest.mark.parametrize("fmt,out_fmt", [("e4m3", "f32"), ("e4m3", "e5m2"), ("e4m3", "bf16"), ("bf16", "fp16"), ("fp16", "e4m3"), ("bf16", "f32")])
@pytest.mark.parametrize("rows,k,cols", SHAPES)
def test_plain_and_residual(op, fmt, out_fmt, rows, k, cols):
    from paper_2303_11257_b200 import lib as L, synth
    fb = "e5m2" if fmt == "e4m3" and op != "fwd" else fmt
    A, B, val, scale = _operands(L, synth, op, rows, k, cols, 61, fmt, fb)
    ws, fn = L.new_workspace(), getattr(L, "us_linear_" + op)
    out = U.empty(rows, cols, out_fmt, PAD(cols))
    fn(A, B, scale, out, ws)
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(out, val, out_fmt, TOL * max(1.0, np.abs(val).max() / 4), f"{op} plain")
    if PAD(cols) > cols:
        assert not out.as_strided((rows, PAD(cols)), (PAD(cols), 1))[:, cols:].contiguous().view(torch.uint8).any()
    for skip_fmt in ("f32", "bf16"):
        sk = synth.normal(61, 2, (rows, cols))
        out = U.empty(rows, cols, out_fmt, PAD(cols))
        fn(A, B, scale, out, ws, L.epilogue(skip=U.to_device(sk, skip_fmt, PAD(cols)), skip_coef=0.8, out_coef=0.6))
        assert L.us_workspace_status(ws) == 0
        ref = O.weighted_add(U.values_of(sk, skip_fmt), val, np.float32(0.8), np.float32(0.6))
        U.assert_close_stored(out, ref, out_fmt, TOL * max(1.0, np.abs(val).max() / 4), f"{op} residual {skip_fmt}")


@pytest.mark.parametrize("fmt,out_fmt", [("e4m3", "e4m3"), ("e4m3", "bf16"), ("bf16", "bf16"), ("fp16", "e5m2")])
@pytest.mark.parametrize("rows,k,cols", [(1, 16, 16), (9, 128, 63), (48, 1024, 400), (129, 304, 97)])
def test_activation_epilogues(fmt, out_fmt, rows, k, cols):
    from paper_2303_11257_b200 import lib as L, synth
    X, W, val, scale = _operands(L, synth, "fwd", rows, k, cols, 62, fmt, fmt)
    ag, bg = S.gelu_scales()
    ws, aux_fmt = L.new_workspace(), "fp16" if fmt == "fp16" else "bf16"
    H, A = U.empty(rows, cols, aux_fmt, PAD(cols)), U.empty(rows, cols, out_fmt, PAD(cols))
    L.us_linear_fwd(X, W, scale, A, ws, L.epilogue(act=L.US_ACT_GELU, act_in_scale=0.9, act_out_scale=float(ag), aux=H))
    U.assert_close_stored(H, val, aux_fmt, TOL, "stored pre-activation")
    U.assert_close_stored(A, O.gelu_fwd(val, 0.9, ag), out_fmt, TOL, "gelu")
    A2 = U.empty(rows, cols, out_fmt, PAD(cols))                       # without the copy of the pre-activation: the same
    L.us_linear_fwd(X, W, scale, A2, ws, L.epilogue(act=L.US_ACT_GELU, act_in_scale=0.9, act_out_scale=float(ag)))
    assert np.array_equal(U.codes_of(A), U.codes_of(A2))
    L.us_linear_fwd(X, W, scale, A, ws, L.epilogue(act=L.US_ACT_TANH, act_in_scale=0.9, act_out_scale=1.5))
    U.assert_close_stored(A, 1.5 * np.tanh(0.9 * val), out_fmt, TOL, "tanh")
    gfmt = "e5m2" if fmt == "e4m3" else fmt
    G, W, val, scale = _operands(L, synth, "bwd_x", rows, k, cols, 63, gfmt, fmt)
    dH = U.empty(rows, cols, out_fmt, PAD(cols))
    L.us_linear_bwd_x(G, W, scale, dH, ws, L.epilogue(act=L.US_ACT_GELU_GRAD, act_in_scale=0.9, act_out_scale=float(bg), aux=H))
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(dH, O.gelu_bwd(U.host_values(H), val, 0.9, bg), out_fmt, TOL, "gelu gradient")


@pytest.mark.parametrize("fmt", ["bf16", "e4m3"])
@pytest.mark.parametrize("rows,k,cols", [(40, 80, 64), (200, 272, 48), (8, 512, 16)])
def test_batched_outputs_of_at_most_64_columns(fmt, rows, k, cols):
    from paper_2303_11257_b200 import lib as L, synth
    n, ws = 6, L.new_workspace()
    for op in ("fwd", "bwd_x", "bwd_w"):
        probs = [_operands(L, synth, op, rows, k, cols, 70 + i, fmt, fmt) for i in range(n)]
        A, B = (torch.stack([p[j].contiguous().view(torch.uint8) for p in probs]).flatten(0, 1).view(U.TORCH_OF[fmt]) for j in (0, 1))
        ra, rb = (A.shape[0] // n, B.shape[0] // n)
        if (A.shape[1] * A.element_size()) % 16 or (B.shape[1] * B.element_size()) % 16:
            continue
        out = U.empty(n * rows, cols, "f32")
        bt = L.batch((2, 3), (3 * ra * A.shape[1], ra * A.shape[1]), (3 * rb * B.shape[1], rb * B.shape[1]), (3 * rows * cols, rows * cols))
        getattr(L, f"us_linear_{op}_batched")(A[:ra], B[:rb], probs[0][3], out[:rows], bt, ws)
        assert L.us_workspace_status(ws) == 0
        for i, p in enumerate(probs):
            U.assert_close_stored(out[i * rows:(i + 1) * rows], p[2], "f32", TOL * max(1.0, np.abs(p[2]).max() / 4), f"{op} problem {i}")


@pytest.mark.parametrize("op,rows,cols", [("bwd_w", 16, 2048), ("bwd_w", 16, 2064), ("bwd_w", 40, 3072), ("bwd_w", 40, 3088), ("bwd_w", 50, 4096), ("bwd_w", 50, 4112),
                                          ("bwd_w", 100, 4112), ("fwd", 7000, 80), ("fwd", 7100, 80)])
@pytest.mark.parametrize("fmt", ["e4m3", "bf16"])
def test_both_sides_of_the_lines_of_the_choice(op, rows, cols, fmt):
    from paper_2303_11257_b200 import lib as L, synth
    A, B, val, scale = _operands(L, synth, op, rows, 144, cols, 64, fmt, fmt)
    ws, out = L.new_workspace(), U.empty(rows, cols, "f32", PAD(cols))
    getattr(L, "us_linear_" + op)(A, B, scale, out, ws)
    assert L.us_workspace_status(ws) == 0
    U.assert_close_stored(out, val, "f32", TOL * max(1.0, np.abs(val).max() / 4), op)
