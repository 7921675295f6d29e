"""us_attention_bwd_all: the whole backward pass of attention in one launch, against the oracle.  dS within one ulp (code) of
the softmax gradient on the unrounded dP; dQ, dK and dV against products of the device's own stored dS and P."""
import numpy as np
import pytest
import torch

from oracle import formats as F
from oracle import ops as O
from tests import util as U

pytestmark = pytest.mark.gpu
TOL = 2e-3


def _run(nb0, nb1, s_q, s_k, fmt, out_fmt, seed, store_ds=True):
    """Separate contiguous tensors of every problem (P and dS with padded rows); results as host values."""
    from paper_2303_11257_b200 import lib as L, synth
    gfmt = "e5m2" if fmt == "e4m3" else fmt
    n = nb0 * nb1
    dc, q, k, v = (synth.normal(seed, i, (n * r, 64)) for i, r in ((0, s_q), (1, s_q), (2, s_k), (3, s_k)))
    dCv, Qv, Kv, Vv = (U.values_of(t, f).reshape(n, -1, 64) for t, f in ((dc, gfmt), (q, fmt), (k, fmt), (v, fmt)))
    ld = (s_k + 15) // 16 * 16
    sm, b_p, b_q, b_k, b_v = float(s_k), 0.125, 0.25, 0.125, s_q ** -0.5
    p_host, _ = O.attention_fwd(Qv, Kv, Vv, 0.125, sm, 1.0, fmt)
    P = U.to_device(p_host.reshape(n * s_q, s_k), fmt, ld)
    dS = U.empty(n * s_q, s_k, gfmt, ld)
    dQ, dK, dV = U.empty(n * s_q, 64, out_fmt), U.empty(n * s_k, 64, out_fmt), U.empty(n * s_k, 64, out_fmt)
    ws = L.new_workspace()
    qs, ks, ps = (nb1 * s_q * 64, s_q * 64), (nb1 * s_k * 64, s_k * 64), (nb1 * s_q * ld, s_q * ld)
    bt = L.attention_bwd_all_batch((nb0, nb1), qs, ps, qs, ks, ks, ps, qs, ks, ks)
    L.us_attention_bwd_all(U.to_device(dc, gfmt)[:s_q], P[:s_q], U.to_device(q, fmt)[:s_q], U.to_device(k, fmt)[:s_k], U.to_device(v, fmt)[:s_k],
                           b_p, sm, sm, b_q, b_k, b_v, dS[:s_q] if store_ds else None, dQ[:s_q], dK[:s_k], dV[:s_k], bt, ws)
    assert L.us_workspace_status(ws) == 0
    return (dCv, Qv, Kv, Vv, p_host), (dS, dQ, dK, dV), (sm, b_p, b_q, b_k, b_v), gfmt


def _close(got, ref, fmt, what):
    lim = TOL * max(1.0, np.abs(ref).max())
    if fmt in ("e4m3", "e5m2"):
        fm = F.FORMATS[fmt]
        ok = (U.code_distance(F.quantise_codes(got, fm), F.quantise_codes(ref, fm), fmt) <= 1) | (np.abs(got - F.quantise(ref, fm)) <= lim)
    else:
        ok = np.abs(got - ref) <= lim + (U.ulp_of(ref, fmt) if fmt != "f32" else 0.0)
    assert ok.all(), f"{what}: {(~ok).sum()} elements out"


# one key and one query; the edges of a query tile, of a key block, of a CTA's 128 keys and of a cluster of two; a last CTA of a cluster
# with one key, none (384 keys or fewer of four CTAs) and all of them; more problems than CTAs (clusters), so that every phase carries over
SHAPES = [(1, 1, 1, 1), (1, 2, 40, 72), (2, 1, 128, 128), (1, 1, 129, 136), (1, 2, 200, 256), (1, 1, 130, 257), (1, 1, 384, 330),
          (1, 2, 512, 512), (3, 60, 136, 200), (2, 40, 264, 272), (5, 20, 130, 64)]


@pytest.mark.parametrize("fmt,out_fmt", [("bf16", "e5m2"), ("fp16", "f32"), ("e4m3", "e5m2"), ("e4m3", "bf16")])
@pytest.mark.parametrize("nb0,nb1,s_q,s_k", SHAPES)
def test_all_gradients_against_the_oracle(nb0, nb1, s_q, s_k, fmt, out_fmt):
    n = nb0 * nb1
    (dC, Q, K, V, p), outs, (sm, b_p, b_q, b_k, b_v), gfmt = _run(nb0, nb1, s_q, s_k, fmt, out_fmt, 31)
    dS, dQ, dK, dV = (U.host_values(t).reshape(n, -1, t.shape[1]) for t in outs)
    dp = b_p * (dC @ V.transpose(0, 2, 1))
    ref = O.softmax_bwd(p, dp, sm, sm)
    tol = 3e-6 * (np.abs(ref).max() + np.abs(dp).max())
    if fmt == "e4m3":
        fm = F.FORMATS[gfmt]
        ok = (U.code_distance(F.quantise_codes(dS, fm), F.quantise_codes(ref, fm), gfmt) <= 1) | (np.abs(dS - F.quantise(ref, fm)) <= tol)
    else:
        ok = np.abs(dS - ref) <= U.ulp_of(ref, fmt) + tol
    assert ok.all(), f"dS: {(~ok).sum()} elements out"
    _close(dQ, b_q * (dS @ K), out_fmt, "dQ")
    _close(dK, b_k * (dS.transpose(0, 2, 1) @ Q), out_fmt, "dK")
    _close(dV, np.float64(np.float32(b_v)) * (p.transpose(0, 2, 1) @ dC), out_fmt, "dV")


@pytest.mark.parametrize("fmt", ["bf16", "e4m3"])
def test_gradients_do_not_depend_on_the_stored_scores_gradient_and_repeat(fmt):
    """dS = None leaves the other results bit for bit; so does a second launch (no atomics)."""
    runs = [_run(2, 45, 200, 400, fmt, "f32", 32, store)[1] for store in (True, True, False)]
    for other in runs[1:]:
        for a, b in zip(runs[0][1:], other[1:]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("s_k", [200, 512])
@pytest.mark.parametrize("fmt", ["bf16", "e4m3"])
def test_long_runs_of_a_cluster(s_k, fmt):
    """Every cluster of two (four) CTAs walks 16 to 50 tiles of 128 queries, so that the area its CTAs exchange parts of dQ in is reused
    as often: dQ against the float64 product of the device's own dS and K, and the same bits from every launch."""
    from paper_2303_11257_b200 import lib as L
    n, s_q, gfmt = 320, 600, "e5m2" if fmt == "e4m3" else fmt
    gen = torch.Generator(device="cuda").manual_seed(33)
    ld = (s_k + 15) // 16 * 16
    rand = lambda r, f: torch.randn(n * r, 64, generator=gen, device="cuda").to(U.TORCH_OF[f])
    dC, Q, K, V = rand(s_q, gfmt), rand(s_q, fmt), rand(s_k, fmt), rand(s_k, fmt)
    P = torch.zeros(n * s_q, ld, device="cuda")
    P[:, :s_k] = s_k * torch.softmax(torch.randn(n * s_q, s_k, generator=gen, device="cuda"), 1)
    P, dS = P.to(U.TORCH_OF[fmt])[:, :s_k], U.empty(n * s_q, s_k, gfmt, ld)
    ws, first = L.new_workspace(), None
    bt = L.attention_bwd_all_batch((1, n), (1, s_q * 64), (1, s_q * ld), (1, s_q * 64), (1, s_k * 64), (1, s_k * 64), (1, s_q * ld), (1, s_q * 64),
                                   (1, s_k * 64), (1, s_k * 64))
    for _ in range(6):
        out = [torch.zeros(n * r, 64, device="cuda") for r in (s_q, s_k, s_k)]
        L.us_attention_bwd_all(dC[:s_q], P[:s_q], Q[:s_q], K[:s_k], V[:s_k], 0.125, s_k, s_k, 0.25, 0.125, 0.5, dS[:s_q], *(t[:r] for t, r in zip(out, (s_q, s_k, s_k))), bt, ws)
        assert L.us_workspace_status(ws) == 0
        first = first or out
        assert all(torch.equal(a, b) for a, b in zip(first, out))
    wide = lambda t, r: t.float().double().reshape(n, r, -1)
    ref = 0.25 * wide(dS, s_q) @ wide(K, s_k)
    assert bool(((first[0].double().reshape(n, s_q, 64) - ref).abs() <= TOL * max(1.0, float(ref.abs().max()))).all())


@pytest.mark.parametrize("fmt,s_k,cl", [("bf16", 100, 1), ("bf16", 200, 2), ("e4m3", 256, 2), ("fp16", 400, 4), ("e4m3", 512, 4)])
def test_a_cluster_that_gives_up_drains_what_its_ctas_send_each_other(fmt, s_k, cl):
    """One CTA of the cluster gets dC for some tiles only: every wait runs out, the status word says so and, with one cluster in the
    launch, nothing else (2 would be stores of a partner that did not come in); the same call without the stall is right afterwards."""
    from paper_2303_11257_b200 import lib as L, synth
    s_q, gfmt, ld = 900, "e5m2" if fmt == "e4m3" else fmt, (s_k + 15) // 16 * 16
    t = lambda i, r, f: U.to_device(synth.normal(34, i, (r, 64)), f)
    dC, Q, K, V = t(0, s_q, gfmt), t(1, s_q, fmt), t(2, s_k, fmt), t(3, s_k, fmt)
    P, dS = U.to_device(np.abs(synth.normal(34, 4, (s_q, s_k))), fmt, ld), U.empty(s_q, s_k, gfmt, ld)
    ws, bt = L.new_workspace(), L.attention_bwd_all_batch((1, 1), *[(1, 1)] * 9)
    call = lambda: [U.empty(r, 64, "f32") for r in (s_q, s_k, s_k)]
    good = call()
    L.us_attention_bwd_all(dC, P, Q, K, V, 1.0, s_k, 1.0, 1.0, 1.0, 1.0, dS, *good, bt, ws)
    assert L.us_workspace_status(ws) == 0
    for rank in range(cl):
        for tile in (0, 1, 2, 3, 5):
            L.us_test_attention_bwd_all_starved(dC, P, Q, K, V, s_k, dS, *call(), bt, ws, wait_limit=2000, rank=rank, tile=tile)
            assert L.us_workspace_status(ws) == 6 and int(ws[:4].view(torch.int32)[0]) == 1, (rank, tile)
            ws.zero_()
    again = call()
    L.us_attention_bwd_all(dC, P, Q, K, V, 1.0, s_k, 1.0, 1.0, 1.0, 1.0, dS, *again, bt, ws)
    assert L.us_workspace_status(ws) == 0 and all(torch.equal(a, b) for a, b in zip(good, again))
    with pytest.raises(L.UnitScaleError) as e:
        L.us_test_attention_bwd_all_starved(dC, P, Q, K, V, s_k, dS, *again, bt, ws, wait_limit=0, rank=0, tile=0)
    assert e.value.status == 1


def _layer(s_q, s_k, fmt, out_fmt, n, seed, spoil=None):
    """(dC, P, Q, K, V), the results' buffers and the two ways to the results, over the layout of an encoder layer: heads are column slices of
    [tokens x 3 x heads x 64] matrices, P and dS have padded rows.  The buffers begin as ones, results' neighbours among them."""
    from paper_2303_11257_b200 import lib as L
    gfmt, h = "e5m2" if fmt == "e4m3" else fmt, 3
    gen = torch.Generator(device="cuda").manual_seed(seed)
    wide = lambda r, f, w: torch.randn(n * r, w * h * 64, generator=gen, device="cuda").to(U.TORCH_OF[f])
    dC, q, kv, ld = wide(s_q, gfmt, 1), wide(s_q, fmt, 1), wide(s_k, fmt, 2), (s_k + 15) // 16 * 16
    P = torch.zeros(n * h * s_q, ld, device="cuda")
    P[:, :s_k] = s_k * torch.softmax(torch.randn(n * h * s_q, s_k, generator=gen, device="cuda"), 1)
    P = P.to(U.TORCH_OF[fmt])[:, :s_k]
    if spoil:
        spoil(dC, kv)
    ones = lambda r, c, f: torch.ones(r, c, device="cuda").to(U.TORCH_OF[f])
    hs = lambda t, r, w, at=0: (t[:r, at * h * 64:at * h * 64 + 64], (r * w * h * 64, 64))       # head 0 of sequence 0, strides
    (dc, sdc), (Q, sq), (K, sk), (V, _) = hs(dC, s_q, 1), hs(q, s_q, 1), hs(kv, s_k, 2), hs(kv, s_k, 2, 1)
    sp, ws = (h * s_q * ld, s_q * ld), L.new_workspace()

    def run(one):
        dS, dq, dkv = ones(n * h * s_q, ld, gfmt)[:, :s_k], ones(n * s_q, h * 64 + 16, out_fmt), ones(n * s_k, 2 * h * 64 + 32, out_fmt)
        dQ, dK, dV = dq[:s_q, :64], dkv[:s_k, :64], dkv[:s_k, h * 64 + 16:h * 64 + 80]
        rq, rk = (s_q * dq.shape[1], 64), (s_k * dkv.shape[1], 64)
        if one:
            L.us_attention_bwd_all(dc, P[:s_q], Q, K, V, 0.125, s_k, s_k, 0.25, 0.125, 0.5, dS[:s_q], dQ, dK, dV,
                                   L.attention_bwd_all_batch((n, h), sdc, sp, sq, sk, sk, sp, rq, rk, rk), ws)
        else:
            L.us_linear_bwd_w_batched(P[:s_q], dc, 0.5, dV, L.batch((n, h), sp, sdc, rk), ws)
            L.us_attention_bwd(dc, P[:s_q], K, V, 0.125, s_k, s_k, 0.25, dS[:s_q], dQ, L.attention_bwd_batch((n, h), sdc, sp, sk, sk, sp, rq), ws)
            L.us_linear_bwd_w_batched(dS[:s_q], Q, 0.125, dK, L.batch((n, h), sp, sq, rk), ws)
        assert L.us_workspace_status(ws) == 0
        return dS, dq, dkv

    return (dC, P, q, kv), run


@pytest.mark.parametrize("s_q,s_k", [(100, 112), (272, 272), (160, 304), (384, 384), (130, 400), (496, 496)])
@pytest.mark.parametrize("fmt,out_fmt", [("bf16", "e5m2"), ("fp16", "f32"), ("e4m3", "bf16")])
def test_strided_heads_and_what_lies_between_them(s_q, s_k, fmt, out_fmt):
    """In the layout of a layer: dS within one code of the three launches' (their row sums have another order), dQ and dK against products of
    the launch's own dS, dV bit for bit that of the batched GEMM; nothing written between the results."""
    n, h = 2, 3
    (dC, P, q, kv), run = _layer(s_q, s_k, fmt, out_fmt, n, 41)
    (dS, dq, dkv), (dS3, dq3, dkv3) = run(True), run(False)
    apart = (dS.float() - dS3.float()).abs()
    # beside one code, 3e-6 of the largest dS and of dP (variance 1, below 16): a float32 difference of the mean where dP is close to it
    tol = 3e-6 * (float(dS3.float().abs().max()) + 16.0)
    assert bool(((apart <= tol).cpu() | torch.from_numpy(U.code_distance(U.codes_of(dS), U.codes_of(dS3), "e5m2" if fmt == "e4m3" else fmt) <= 1)).all())
    pieces = lambda t, s, at: t.float().double().reshape(n, s, -1)[:, :, at:at + h * 64].reshape(n, s, h, 64).transpose(1, 2).cpu().numpy()
    w = dS.float().double().reshape(n, h, s_q, s_k).cpu().numpy()
    _close(pieces(dq, s_q, 0), 0.25 * w @ pieces(kv, s_k, 0), out_fmt, "dQ")
    _close(pieces(dkv, s_k, 0), 0.125 * w.transpose(0, 1, 3, 2) @ pieces(q, s_q, 0), out_fmt, "dK")
    at = h * 64 + 16
    assert torch.equal(dkv[:, at:at + h * 64].contiguous().view(torch.uint8), dkv3[:, at:at + h * 64].contiguous().view(torch.uint8))
    for t, gaps in ((dq, [slice(h * 64, None)]), (dkv, [slice(h * 64, at), slice(at + h * 64, None)])):
        assert all(bool((t[:, g].float() == 1).all()) for g in gaps)


@pytest.mark.parametrize("s_q,s_k", [(100, 100), (300, 208), (200, 336)])
@pytest.mark.parametrize("fmt", ["bf16", "e4m3"])
@pytest.mark.parametrize("what", ["inf in dC", "nan in dC", "nan in V", "nan in K"])
def test_gradients_that_are_not_finite_spread_as_with_three_launches(s_q, s_k, fmt, what):
    if fmt == "e4m3" and s_k % 16:
        s_k = 112                                                        # FP8 rows of P start on 16 bytes
    def spoil(dC, kv):
        if what.endswith("dC"):
            dC[37, 70] = float("inf") if what[0] == "i" else float("nan")           # sequence 0, head 1
        else:
            kv[s_k + 5, (3 if what.endswith("V") else 0) * 64 + 130] = float("nan")  # sequence 1, head 2
    _, run = _layer(s_q, s_k, fmt, "f32", 2, 42, spoil)
    finite = [[torch.isfinite(t.float()) for t in run(one)] for one in (True, False)]
    assert not all(bool(t.all()) for t in finite[1]) and all(bool(t.any()) for t in finite[1])
    assert all(torch.equal(a, b) for a, b in zip(*finite))
