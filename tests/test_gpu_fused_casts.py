"""Results that leave their producer in FP8 as well: the copy is, code for code, what us_cast_fp8 makes of the stored result, and the
result is what the call without a copy stores."""
import numpy as np
import pytest
import torch

from tests import util as U

pytestmark = pytest.mark.gpu
PAD = lambda c: (c + 15) // 16 * 16


def _check(L, got, copy, want):
    assert torch.equal(got.contiguous().view(torch.uint8), want.contiguous().view(torch.uint8))
    q = torch.zeros_like(copy.contiguous().view(torch.uint8)).view(copy.dtype)
    L.us_cast_fp8(got, 1.0, q)
    assert np.array_equal(U.codes_of(copy), U.codes_of(q))
    if copy.stride(0) > copy.shape[1]:                                 # nothing behind the rows' ends
        assert not copy.as_strided((copy.shape[0], copy.stride(0)), (copy.stride(0), 1)).view(torch.uint8)[:, copy.shape[1]:].any()


def _call(L, name, *args):
    L._check(name, L._entry(name)(*args, L.current_stream()))


# a narrow tile, one 128 x 128 tile and its ragged end, pair tiles; row pitches on 32-byte boundaries and not
@pytest.mark.parametrize("b,m,n", [(1, 16, 16), (40, 144, 33), (129, 272, 81), (1000, 400, 1040), (2600, 80, 1063)])
@pytest.mark.parametrize("out,q,skip", [("bf16", "e4m3", "f32"), ("f32", "e5m2", "bf16"), ("fp16", "e4m3", "fp16")])
def test_residual_gemm_and_group(b, m, n, out, q, skip):
    from paper_2303_11257_b200 import lib as L, synth
    ws, dev = L.new_workspace(), lambda i, s, f: U.to_device(300.0 * synth.normal(5, i, s) if i == 2 else synth.normal(5, i, s), f, PAD(s[1]))
    X, W, S = dev(0, (b, m), "e4m3"), dev(1, (m, n), "e4m3"), dev(2, (b, n), skip)      # some results beyond E4M3's range
    ep = L.epilogue(skip=S, skip_coef=0.8, out_coef=0.6)
    Y, Y0, Yq = U.empty(b, n, out, PAD(n)), U.empty(b, n, out, PAD(n)), U.empty(b, n, q, PAD(n))
    L.us_linear_fwd(X, W, m ** -0.5, Y0, ws, ep)
    _call(L, "us_linear_fwd_cast", X, W, m ** -0.5, ep, Y, Yq, ws, ws)
    _check(L, Y, Yq, Y0)
    G = dev(3, (b, n), "e5m2")
    dW, dW0, Z, Zq = U.empty(m, n, "f32", PAD(n)), U.empty(m, n, "f32", PAD(n)), U.empty(b, n, out, PAD(n)), U.empty(b, n, q, PAD(n))
    calls = (L.us_linear_call * 2)(L.linear_call(L.US_OP_BWD_W, X, G, 0.1, dW), L.linear_call(L.US_OP_FWD, X, W, m ** -0.5, Z, ep))
    _call(L, "us_linear_group_cast", 2, calls, (L.us_mat * 2)(L.us_mat(), L.mat(Zq)), ws, ws)
    _check(L, Z, Zq, Y0)
    L.us_linear_bwd_w(X, G, 0.1, dW0, ws)
    assert torch.equal(dW, dW0) and L.us_workspace_status(ws) == 0


@pytest.mark.parametrize("rows,cols", [(1, 8), (37, 100), (700, 1024), (300, 1600), (50, 2304)])
@pytest.mark.parametrize("x,out,q", [("bf16", "bf16", "e4m3"), ("fp16", "f32", "e5m2"), ("f32", "fp16", "e5m2")])
def test_layer_norm(rows, cols, x, out, q):
    from paper_2303_11257_b200 import lib as L, synth
    X, w, c = U.to_device(synth.normal(6, 0, (rows, cols)), x), U.to_device(200.0 * synth.normal(6, 1, (1, cols)), "f32"), U.to_device(synth.normal(6, 2, (1, cols)), "f32")
    Y, Y0, Yq = U.empty(rows, cols, out), U.empty(rows, cols, out), U.empty(rows, cols, q)
    L.us_layer_norm_fwd(X, w[0], c[0], 1e-5, Y0)
    _call(L, "us_layer_norm_fwd_cast", X, w, c, 1e-5, Y, Yq)
    _check(L, Y, Yq, Y0)
    G = U.to_device(synth.normal(6, 3, (rows, cols)), x if x != "fp16" else "f32")
    dw, dc, dw0, dc0 = (torch.empty(1, cols, device="cuda") for _ in range(4))
    ws = torch.empty(max(16, L.us_layer_norm_bwd_workspace_bytes(rows, cols)), dtype=torch.uint8, device="cuda")
    L.us_layer_norm_bwd(X, w[0], G, 1e-5, 1.0, 0.5, Y0, dw0[0], dc0[0], ws)
    _call(L, "us_layer_norm_bwd_cast", X, w, G, 1e-5, 1.0, 0.5, Y, Yq, dw, dc, ws, ws)
    _check(L, Y, Yq, Y0)
    assert torch.equal(dw, dw0) and torch.equal(dc, dc0)


def test_a_refused_group_makes_its_copies_by_casts():
    """More tiles than the work list holds: the prepared group goes out as single launches, and the copy as a cast."""
    from paper_2303_11257_b200 import lib as L, synth
    n, k, ws = 46 * 256, 16, L.new_workspace()
    X, W = (U.to_device(synth.normal(60, i, s), "e4m3") for i, s in ((0, (n, k)), (1, (k, n))))
    Y, Yq = U.empty(n, n, "bf16"), U.empty(n, n, "e5m2")
    call = L.Plan((), ()).group([(L.US_OP_FWD, X, W, 0.25, Y, Y, (0.0, 1.0))], ws, {0: Yq})
    call(L.current_stream())
    assert call.refused
    q = U.empty(n, n, "e5m2")
    L.us_cast_fp8(Y, 1.0, q)
    assert L.us_workspace_status(ws) == 0 and torch.equal(Yq.view(torch.uint8), q.view(torch.uint8)) and bool(q.view(torch.uint8).any())
