"""us_layer_norm_fwd / us_layer_norm_bwd against the oracle."""
import numpy as np
import pytest
import torch

from oracle import formats as F
from oracle import ops as O
from tests import util as U

pytestmark = pytest.mark.gpu


def _lib():
    from paper_2303_11257_b200 import lib
    return lib


def _inputs(seed, rows, cols, x_fmt, shift=0.5, spread=1.5):
    from paper_2303_11257_b200 import synth
    X = synth.normal(seed, 0, (rows, cols), spread) + np.float32(shift)
    G = synth.normal(seed, 1, (rows, cols), 1.0)
    w = (1 + 0.25 * synth.normal(seed, 2, (1, cols), 1.0)).astype(np.float32)
    c = (0.1 * synth.normal(seed, 3, (1, cols), 1.0)).astype(np.float32)
    if x_fmt != "f32":
        X = F.quantise(X, F.FORMATS[x_fmt]).astype(np.float32)
        G = F.quantise(G, F.FORMATS[x_fmt]).astype(np.float32)
    return X, G, w, c


CASES = [(1, 8, "f32", None), (5, 24, "f32", None), (33, 100, "f32", None), (64, 256, "bf16", None), (130, 768, "bf16", 800),
         (257, 1024, "bf16", None), (19, 1000, "fp16", 1008), (40, 2048, "bf16", None), (9, 4096, "f32", None), (6, 2056, "bf16", None)]


@pytest.mark.parametrize("rows,cols,x_fmt,ld", CASES)
@pytest.mark.parametrize("out_fmt", ["f32", "bf16", "e4m3"])
def test_layer_norm_forward(rows, cols, x_fmt, ld, out_fmt):
    L = _lib()
    X, _, w, c = _inputs(3, rows, cols, x_fmt)
    eps = 1e-5
    Y = U.empty(rows, cols, out_fmt, ld)
    L.us_layer_norm_fwd(U.to_device(X, x_fmt, ld), torch.from_numpy(w[0]).cuda(), torch.from_numpy(c[0]).cuda(), eps, Y)
    ref = O.layer_norm_fwd(X, w, c, np.float32(eps))
    # float32 arithmetic on O(1) values with sums over up to 4096 elements: 2e-5 absolute before the output rounding
    U.assert_close_stored(Y, ref, out_fmt, 2e-5)


@pytest.mark.parametrize("rows,cols,x_fmt,ld", CASES)
def test_layer_norm_backward(rows, cols, x_fmt, ld):
    L = _lib()
    X, G, w, _ = _inputs(4, rows, cols, x_fmt)
    eps, beta_x, beta_wc = 1e-5, 1.0, float(np.float32(rows ** -0.5))
    dX = U.empty(rows, cols, "f32", ld)
    dw = torch.empty(cols, device="cuda")
    dc = torch.empty(cols, device="cuda")
    ws = torch.empty(max(L.us_layer_norm_bwd_workspace_bytes(rows, cols), 16), dtype=torch.uint8, device="cuda")
    args = (U.to_device(X, x_fmt, ld), torch.from_numpy(w[0]).cuda(), U.to_device(G, x_fmt, ld), eps, beta_x, beta_wc)
    L.us_layer_norm_bwd(*args, dX, dw, dc, ws)
    rdX, rdw, rdc = O.layer_norm_bwd(X, w, G, np.float32(eps), beta_x, beta_wc)
    scale = 1.0 / np.sqrt(X.var(axis=1).min() + eps)          # dX grows with 1 / sigma
    assert np.abs(U.host_values(dX) - rdX).max() <= 3e-5 * max(1.0, scale)
    # column sums of `rows` products of O(1) values in float32, scaled by rows^-1/2
    tol = 2e-6 * np.sqrt(rows) + 1e-6
    assert np.abs(dw.cpu().numpy() - rdw.reshape(-1)).max() <= tol * 8
    assert np.abs(dc.cpu().numpy() - rdc.reshape(-1)).max() <= tol * 8
    # a second call gives bit-identical results (fixed summation order)
    dX2, dw2, dc2 = U.empty(rows, cols, "f32", ld), torch.empty_like(dw), torch.empty_like(dc)
    L.us_layer_norm_bwd(*args, dX2, dw2, dc2, ws)
    assert torch.equal(dw, dw2) and torch.equal(dc, dc2) and torch.equal(dX.contiguous(), dX2.contiguous())


def test_layer_norm_large_offset_rows_keep_their_variance():
    """Rows with a mean far above their spread: the variance about the mean survives float32
    (mean(x^2) - mu^2 in float32 would not)."""
    L = _lib()
    X, _, w, c = _inputs(5, 16, 1024, "f32", shift=300.0, spread=0.5)
    Y = U.empty(16, 1024, "f32")
    L.us_layer_norm_fwd(torch.from_numpy(X).cuda(), torch.from_numpy(w[0]).cuda(), torch.from_numpy(c[0]).cuda(), 0.0, Y)
    assert np.abs(U.host_values(Y) - O.layer_norm_fwd(X, w, c, 0.0)).max() < 5e-4      # input ulp 3e-5 / sigma 0.5


def test_layer_norm_errors_and_empty():
    L = _lib()
    x = torch.zeros((4, 16), device="cuda")
    v = torch.ones(16, device="cuda")
    with pytest.raises(L.UnitScaleError) as e:
        L.us_layer_norm_fwd(x, torch.ones(8, device="cuda"), v, 0.0, torch.empty_like(x))
    assert e.value.status == 1
    with pytest.raises(L.UnitScaleError) as e:
        L.us_layer_norm_fwd(x, v, v, -1.0, torch.empty_like(x))
    assert e.value.status == 1
    ws = torch.empty(16, dtype=torch.uint8, device="cuda")
    with pytest.raises(L.UnitScaleError) as e:                       # workspace too small
        L.us_layer_norm_bwd(x, v, x, 0.0, 1.0, 0.5, torch.empty_like(x), torch.empty_like(v), torch.empty_like(v), ws)
    assert e.value.status == 4
    big = torch.zeros((2, 4104), device="cuda")
    vb = torch.ones(4104, device="cuda")
    wsb = torch.empty(L.us_layer_norm_bwd_workspace_bytes(2, 4104), dtype=torch.uint8, device="cuda")
    with pytest.raises(L.UnitScaleError) as e:                       # rows longer than the backward supports
        L.us_layer_norm_bwd(big, vb, big, 0.0, 1.0, 0.5, torch.empty_like(big), torch.empty_like(vb), torch.empty_like(vb), wsb)
    assert e.value.status == 2
    L.us_layer_norm_fwd(torch.zeros((0, 16), device="cuda"), v, v, 0.0, torch.zeros((0, 16), device="cuda"))


@pytest.mark.parametrize("rows,cols,ld", [(64, 256, None), (130, 768, 800), (257, 1024, None), (40, 512, None)])
def test_layer_norm_backward_with_a_float32_gradient(rows, cols, ld):
    """16-bit X with a float32 incoming gradient (the gradient of a layer's output)."""
    L = _lib()
    X, G, w, _ = _inputs(6, rows, cols, "bf16")
    from paper_2303_11257_b200 import synth
    G = synth.normal(6, 4, (rows, cols), 1.0)                      # not on the BF16 grid
    eps, beta_wc = 1e-5, float(np.float32(rows ** -0.5))
    dX, dw, dc = U.empty(rows, cols, "bf16", ld), torch.empty(cols, device="cuda"), torch.empty(cols, device="cuda")
    ws = torch.empty(L.us_layer_norm_bwd_workspace_bytes(rows, cols), dtype=torch.uint8, device="cuda")
    L.us_layer_norm_bwd(U.to_device(X, "bf16", ld), torch.from_numpy(w[0]).cuda(), U.to_device(G, "f32", ld), eps, 1.0, beta_wc,
                        dX, dw, dc, ws)
    rdX, rdw, rdc = O.layer_norm_bwd(X, w, G, np.float32(eps), 1.0, beta_wc)
    scale = 1.0 / np.sqrt(X.var(axis=1).min() + eps)
    U.assert_close_stored(dX, rdX, "bf16", 3e-5 * max(1.0, scale), "dX")
    tol = 8 * (2e-6 * np.sqrt(rows) + 1e-6)
    assert np.abs(dw.cpu().numpy() - rdw.reshape(-1)).max() <= tol and np.abs(dc.cpu().numpy() - rdc.reshape(-1)).max() <= tol


@pytest.mark.parametrize("x_fmt,g_fmt,out_fmt,q_fmt", [("bf16", "bf16", "bf16", "e5m2"), ("fp16", "f32", "fp16", "e4m3"), ("bf16", "f32", "f32", None), ("fp16", "fp16", "bf16", "e5m2")])
@pytest.mark.parametrize("rows,cols", [(1, 8), (3, 264), (37, 256), (130, 776), (67, 1288), (9, 2048), (5000, 136)])
def test_layer_norm_backward_with_rows_among_several_warps(rows, cols, x_fmt, g_fmt, out_fmt, q_fmt):
    """Rows of one to eight warps, turns of one to four rows, every output kind: dX and its copy in FP8, dw and dc."""
    from paper_2303_11257_b200 import lib as L, synth
    X, G, w, _ = _inputs(8, rows, cols, x_fmt)
    G = synth.normal(8, 4, (rows, cols), 1.0)
    eps, beta_wc = 1e-5, float(np.float32(rows ** -0.5))
    dX, q = U.empty(rows, cols, out_fmt, cols + 24), U.empty(rows, cols, q_fmt, cols + 8) if q_fmt else None
    dw, dc = torch.empty(cols, device="cuda"), torch.empty(cols, device="cuda")
    ws = torch.empty(max(16, L.us_layer_norm_bwd_workspace_bytes(rows, cols)), dtype=torch.uint8, device="cuda")
    args = (U.to_device(X, x_fmt), U.to_device(w, "f32"), U.to_device(G, g_fmt))
    tail = (L._vec(dw), L._vec(dc), ws.data_ptr(), ws.numel())
    m = [L.mat(t) for t in (*args, dX)]
    name = "us_layer_norm_bwd_cast" if q_fmt else "us_layer_norm_bwd"
    L.Call(name, m[0], m[1], m[2], eps, 1.0, beta_wc, m[3], *([L.mat(q)] if q_fmt else []), *tail)(L.current_stream())
    Xv, Gv = U.values_of(X, x_fmt), U.values_of(G, g_fmt)
    rx, rw, rc = O.layer_norm_bwd(Xv, w.astype(np.float64), Gv, eps, 1.0, beta_wc)
    scale = 1.0 / np.sqrt(Xv.var(axis=1).min() + eps)
    U.assert_close_stored(dX, rx, out_fmt, 3e-5 * max(1.0, scale), "dX")
    tol = 8 * (2e-6 * np.sqrt(rows) + 1e-6)
    assert np.abs(U.host_values(dw) - rw.ravel()).max() <= tol and np.abs(U.host_values(dc) - rc.ravel()).max() <= tol
    if q_fmt:
        most = 448 if q_fmt == "e4m3" else 57344
        assert torch.equal(q.contiguous().view(torch.uint8), dX.float().clamp(-most, most).to(U.TORCH_OF[q_fmt]).contiguous().view(torch.uint8))


@pytest.mark.parametrize("cols", [512, 1024, 2048])
@pytest.mark.parametrize("g_fmt", ["fp16", "f32"])
def test_layer_norm_backward_of_rows_far_from_zero(cols, g_fmt):
    """Rows of whole numbers about 1500 with a spread of 1.4 and a gradient that goes along with them: sums and means are exact in float32, so
    that x - mu is.  What is left is 1 / sigma and the products: 2^-22 relative in every term of dX (at most 8 of up to 4), and in the 16
    terms of dw.  (A normalised input formed as x / sigma - mu / sigma rounds at 1060: 6e-5 in dX, 8e-4 in dw.)"""
    from paper_2303_11257_b200 import lib as L
    rows, rng = 16, np.random.default_rng(cols)
    D = rng.integers(-2, 3, (rows, cols))
    X, G, w = (1500 + D).astype(np.float32), (1 + D + rng.integers(-1, 2, (rows, cols))).astype(np.float32), np.ones((1, cols), np.float32)
    dX, dw, dc = U.empty(rows, cols, "f32"), torch.empty(cols, device="cuda"), torch.empty(cols, device="cuda")
    ws = torch.empty(max(L.us_layer_norm_bwd_workspace_bytes(rows, cols), 16), dtype=torch.uint8, device="cuda")
    L.us_layer_norm_bwd(U.to_device(X, "fp16"), torch.from_numpy(w[0]).cuda(), U.to_device(G, g_fmt), 1e-5, 1.0, 1.0, dX, dw, dc, ws)
    rdX, rdw, rdc = O.layer_norm_bwd(X, w, G, np.float32(1e-5), 1.0, 1.0)
    assert np.abs(U.host_values(dX) - rdX).max() <= 1e-5
    assert np.abs(dw.cpu().numpy() - rdw.reshape(-1)).max() <= 5e-5
    assert np.array_equal(dc.cpu().numpy(), rdc.reshape(-1).astype(np.float32))


@pytest.mark.parametrize("rows,cols", [(37, 256), (70, 1000), (70, 1536), (300, 2048)])
@pytest.mark.parametrize("g_fmt", ["bf16", "f32"])
def test_layer_norm_backward_of_rows_that_are_not_finite(rows, cols, g_fmt):
    """A NaN or an infinity makes its own row of dX NaN and no other; a row whose squares overflow float32 has 1 / sigma = 0 and a gradient of 0."""
    from paper_2303_11257_b200 import lib as L
    X, G, w, _ = _inputs(10, rows, cols, "bf16")
    bad = [5, rows // 2, rows - 1]
    for r, v in zip(bad, (np.nan, np.inf, -np.inf)):
        X[r, cols // 3] = v
    X[7] = np.float32(2.0 ** 70) * np.where(np.arange(cols) % 3, 1, -1)
    dX, dw, dc = U.empty(rows, cols, "f32"), torch.empty(cols, device="cuda"), torch.empty(cols, device="cuda")
    ws = torch.empty(max(L.us_layer_norm_bwd_workspace_bytes(rows, cols), 16), dtype=torch.uint8, device="cuda")
    Xt = torch.from_numpy(X).cuda().bfloat16()
    L.us_layer_norm_bwd(Xt, torch.from_numpy(w[0]).cuda(), U.to_device(G, g_fmt), 1e-5, 1.0, 1.0, dX, dw, dc, ws)
    got, good = dX.cpu().numpy(), np.setdiff1d(np.arange(rows), bad + [7])
    assert np.isnan(got[bad]).all() and not got[7].any()
    ref = O.layer_norm_bwd(X[good], w, G[good], np.float32(1e-5), 1.0, 1.0)[0]
    assert np.abs(got[good] - ref).max() <= 3e-5 * max(1.0, 1.0 / np.sqrt(X[good].var(axis=1).min() + 1e-5))


@pytest.mark.parametrize("rows,cols", [(1, 2048), (60, 2048), (300, 128), (200, 1288), (1000, 768), (5000, 136)])
def test_layer_norm_backward_workspace_of_one_partial_row_per_eight_or_four_rows(rows, cols):
    """The workspace is a row of 2 x cols partial sums per CTA of the widest grid: rows / 8 up to two per SM, or rows / 4 up to three.  A
    buffer of that size is enough and nothing is written beyond it; a smaller one is refused."""
    L = _lib()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    need = 8 * cols * max(min(-(-rows // 8), 2 * sms), min(-(-rows // 4), 3 * sms))
    assert L.us_layer_norm_bwd_workspace_bytes(rows, cols) == need
    X, G, w, _ = _inputs(9, rows, cols, "bf16")
    dX, dw, dc = U.empty(rows, cols, "f32"), torch.empty(cols, device="cuda"), torch.empty(cols, device="cuda")
    buf = torch.full((need + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    args = (U.to_device(X, "bf16"), torch.from_numpy(w[0]).cuda(), U.to_device(G, "bf16"), 1e-5, 1.0, 1.0, dX, dw, dc)
    L.us_layer_norm_bwd(*args, buf[:need])
    rdX, rdw, rdc = O.layer_norm_bwd(X, w, G, np.float32(1e-5), 1.0, 1.0)
    assert (buf[need:] == 0xA5).all()
    assert np.abs(U.host_values(dX) - rdX).max() <= 3e-5 * max(1.0, 1.0 / np.sqrt(X.var(axis=1).min() + 1e-5))
    tol = 8 * (2e-6 * np.sqrt(rows) + 1e-6) * np.sqrt(rows)
    assert np.abs(dw.cpu().numpy() - rdw.reshape(-1)).max() <= tol and np.abs(dc.cpu().numpy() - rdc.reshape(-1)).max() <= tol
    with pytest.raises(L.UnitScaleError) as e:
        L.us_layer_norm_bwd(*args, buf[:need - 16])
    assert e.value.status == L.US_ERR_WORKSPACE


@pytest.mark.parametrize("rows,cols,q_fmt", [(16400, 1024, None), (16384, 896, "e4m3"), (12289, 640, "e5m2"), (33000, 512, None), (12000, 640, "e5m2")])
def test_layer_norm_backward_beyond_what_l2_holds(rows, cols, q_fmt):
    """The warp-per-row kernel with its ring of bulk copies, several rows a slot, and its FP8 copy (the last shape is on the other side of
    the line): all of dX, dw and dc against float64."""
    from paper_2303_11257_b200 import lib as L
    torch.manual_seed(rows)
    X, G = (torch.randn(rows, cols, device="cuda") * 1.5 + 0.5).bfloat16(), torch.randn(rows, cols, device="cuda").bfloat16()
    w = 1 + 0.25 * torch.randn(1, cols, device="cuda")
    dX, q = torch.empty_like(X), U.empty(rows, cols, q_fmt) if q_fmt else None
    dw, dc = torch.empty(1, cols, device="cuda"), torch.empty(1, cols, device="cuda")
    ws = torch.empty(L.us_layer_norm_bwd_workspace_bytes(rows, cols), dtype=torch.uint8, device="cuda")
    name, bw = ("us_layer_norm_bwd_cast" if q_fmt else "us_layer_norm_bwd"), rows ** -0.5
    m = [L.mat(t) for t in (X, w, G, dX)]
    L.Call(name, *m[:3], 1e-5, 1.0, bw, m[3], *([L.mat(q)] if q_fmt else []), L.mat(dw), L.mat(dc), ws.data_ptr(), ws.numel())(L.current_stream())
    x, g, u = X.double(), G.double(), G.double() * w.double()
    d = x - x.mean(1, keepdim=True)
    r = (d.square().mean(1, keepdim=True) + 1e-5).rsqrt()
    ref = r * (u - u.mean(1, keepdim=True) - d * r * (u * d * r).mean(1, keepdim=True))
    assert ((dX.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 3e-5).all()             # half a BF16 step, rounded up, and float32 sums
    tol = 8 * (2e-6 * rows ** 0.5 + 1e-6)
    assert (dw.double() - bw * (g * d * r).sum(0)).abs().max() <= tol and (dc.double() - bw * g.sum(0)).abs().max() <= tol
    if q_fmt:
        most = 448 if q_fmt == "e4m3" else 57344
        assert torch.equal(q.view(torch.uint8), dX.float().clamp(-most, most).to(U.TORCH_OF[q_fmt]).view(torch.uint8))
