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


# one key and one query; the edges of a query tile, of a key block, of a 128-key half and of a CTA's 256 keys; the partner CTA with
# one key, an odd number of blocks and all of them; more problems than CTAs (clusters), so that every phase carries over
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
