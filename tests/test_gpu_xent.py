"""us_softmax_xent_fwd / us_softmax_xent_bwd against the oracle.  exp and log go through ex2.approx /
lg2.approx in float32: 2e-6 relative to the row's score range for the log-likelihood, 3e-6 * beta * |g|
for the gradient, plus the rounding of the output format."""
import numpy as np
import pytest
import torch

from oracle import ops as O
from oracle import scales as S
from tests import util as U

pytestmark = pytest.mark.gpu


def _mods():
    from paper_2303_11257_b200 import lib, synth
    return lib, synth


@pytest.mark.parametrize("shape,ld", [((1, 8), None), ((5, 7), None), ((33, 512), None), ((130, 200), 208), ((9, 2048), None),
                                      ((4, 2056), None), ((3, 30522), None)])
@pytest.mark.parametrize("in_fmt,out_fmt", [("f32", "f32"), ("bf16", "bf16"), ("fp16", "e5m2")])
def test_softmax_xent_fwd_bwd(shape, ld, in_fmt, out_fmt):
    L, synth = _mods()
    rows, s = shape
    x = synth.normal(31, 0, shape, 2.0)
    rng = np.random.default_rng(31)
    t = rng.integers(0, s, rows).astype(np.int32)
    g = synth.normal(31, 1, (1, rows))[0]
    beta = S.softmax_xent_scales(s)[1] if s > 1 else 1.0
    Xt = U.to_device(x, in_fmt, ld)
    xv = U.values_of(x, in_fmt)
    tt, gt = torch.from_numpy(t).cuda(), torch.from_numpy(g).cuda()
    out = torch.empty(rows, device="cuda")
    L.us_softmax_xent_fwd(Xt, tt, out)
    ref = O.softmax_xent_fwd(xv, t)
    assert np.abs(out.cpu().numpy() - ref).max() <= 4e-6 * (1 + np.abs(ref).max())
    dX = U.empty(rows, s, out_fmt, ld)
    L.us_softmax_xent_bwd(Xt, tt, gt, beta, dX)
    refb = O.softmax_xent_bwd(xv, t, g.astype(np.float64), beta)
    U.assert_close_stored(dX, refb, out_fmt, 3e-6 * beta * np.abs(g).max(), "xent bwd")
    # g = NULL means ones
    L.us_softmax_xent_bwd(Xt, tt, None, beta, dX)
    U.assert_close_stored(dX, O.softmax_xent_bwd(xv, t, np.ones(rows), beta), out_fmt, 3e-6 * beta, "xent bwd, unit g")


def test_softmax_xent_unit_scale_and_bad_targets():
    L, synth = _mods()
    rows, s = 512, 4096
    X = torch.from_numpy(synth.normal(32, 0, (rows, s), 0.01)).cuda()
    t = torch.from_numpy(np.random.default_rng(32).integers(0, s, rows).astype(np.int32)).cuda()
    dX = torch.empty_like(X)
    L.us_softmax_xent_bwd(X, t, None, S.softmax_xent_scales(s)[1], dX)
    assert abs(dX.pow(2).mean().sqrt().item() - 1) < 0.01            # table row: beta = s / sqrt(s - 1)
    assert dX.sum(dim=1).abs().max().item() < 1e-3
    bad = t.clone(); bad[3] = s; bad[5] = -1
    out = torch.empty(rows, device="cuda")
    L.us_softmax_xent_fwd(X, bad, out)
    assert torch.isnan(out[[3, 5]]).all() and torch.isfinite(out[[0, 1, 2, 4]]).all()
    L.us_softmax_xent_bwd(X, bad, None, 1.0, dX)
    assert (dX[3] < 0).all() and (dX[5] < 0).all()                    # no one-hot term: -softmax only
    with pytest.raises(L.UnitScaleError) as e:
        L.us_softmax_xent_bwd(X, t, None, 1.0, torch.empty((rows, s + 8), device="cuda"))
    assert e.value.status == 1


# Class counts at the edges of the row kernel's choices: a warp per row up to 512, then 128 ... 1024 threads with 1 to 8
# (float32: 4) chunks of eight per thread, then rows that are re-read; row ends inside a chunk, with and without an
# aligned row pitch.
@pytest.mark.parametrize("cols", [512, 513, 1023, 1025, 4097, 8192, 8193, 16391, 30522, 30527, 32768, 32769, 36000, 36001, 65536, 65541])
@pytest.mark.parametrize("in_fmt,out_fmt,pad", [("bf16", "e5m2", True), ("fp16", "f32", False), ("f32", "bf16", True)])
def test_softmax_xent_row_kernel_edges(cols, in_fmt, out_fmt, pad):
    L, synth = _mods()
    rows, ld = 3, ((cols + 15) // 16 * 16 if pad else None)
    x = synth.normal(33, cols, (rows, cols), 2.0)
    x[1, 5:9] = -np.inf                                               # masked classes
    t = np.array([0, cols - 1, cols // 2], np.int32)
    Xt, xv = U.to_device(x, in_fmt, ld), U.values_of(x, in_fmt)
    tt = torch.from_numpy(t).cuda()
    out, dX = torch.empty(rows, device="cuda"), U.empty(rows, cols, out_fmt, ld)
    L.us_softmax_xent_fwd(Xt, tt, out)
    ref = O.softmax_xent_fwd(xv, t)
    assert np.abs(out.cpu().numpy() - ref).max() <= 4e-6 * (1 + np.abs(ref).max())
    L.us_softmax_xent_bwd(Xt, tt, None, 8.0, dX)
    U.assert_close_stored(dX, O.softmax_xent_bwd(xv, t, np.ones(rows), 8.0), out_fmt, 3e-6 * 8.0, "xent bwd")


# The forward pass of many rows: a warp per row up to 1280 classes from 16 rows per SM and 4 rows per class on (16-bit: 1536 from 10 rows per class), and the row
# kernel right beside that line.
@pytest.mark.parametrize("rows,cols", [(2368, 513), (2367, 513), (2400, 595), (4096, 1024), (4095, 1024), (5120, 1280), (5121, 1275), (5124, 1281), (14060, 1406), (14059, 1406)])
@pytest.mark.parametrize("in_fmt", ["bf16", "fp16", "f32"])
def test_softmax_xent_forward_of_many_rows(rows, cols, in_fmt):
    L, synth = _mods()
    x = synth.normal(34, cols, (rows, cols), 2.0)
    t = (np.arange(rows) * 7919 % cols).astype(np.int32)
    out = torch.empty(rows, device="cuda")
    L.us_softmax_xent_fwd(U.to_device(x, in_fmt, (cols + 15) // 16 * 16), torch.from_numpy(t).cuda(), out)
    ref = O.softmax_xent_fwd(U.values_of(x, in_fmt), t)
    assert np.abs(out.cpu().numpy() - ref).max() <= 4e-6 * (1 + np.abs(ref).max())


@pytest.mark.parametrize("rows,cols", [(2400, 4104), (2400, 8192), (1300, 8201), (1000, 16384), (2400, 5003), (1300, 10249), (1200, 16384)])
@pytest.mark.parametrize("in_fmt,out_fmt", [("bf16", "e5m2"), ("fp16", "bf16")])
def test_softmax_xent_backward_of_rows_that_a_cta_walks(rows, cols, in_fmt, out_fmt):
    """16-bit rows of 4097 to 16384 classes: CTAs that walk four or more rows through their ring of three, at both CTA sizes and with
    ragged ends (5000 to 8192 classes and from 10241 on; the other two sizes take the register form), with targets outside the row and a
    gradient per row; every 37th row and the last ones against the oracle."""
    L, synth = _mods()
    ld = (cols + 15) // 16 * 16
    x, g = synth.normal(35, cols, (rows, cols), 2.0), synth.normal(35, 1, (1, rows))[0]
    t = (np.arange(rows) * 7919 % cols).astype(np.int32)
    t[37], t[74] = -1, cols
    Xt, xv, dX = U.to_device(x, in_fmt, ld), U.values_of(x, in_fmt), U.empty(rows, cols, out_fmt, ld)
    L.us_softmax_xent_bwd(Xt, torch.from_numpy(t).cuda(), torch.from_numpy(g).cuda(), 8.0, dX)
    pick = np.unique(np.concatenate([np.arange(0, rows, 37), np.arange(rows - 5, rows)]))
    ref = O.softmax_xent_bwd(xv[pick], np.clip(t[pick], 0, cols - 1), g[pick].astype(np.float64), 8.0)
    for i in np.flatnonzero((t[pick] < 0) | (t[pick] >= cols)):       # no one-hot term there
        ref[i, np.clip(t[pick[i]], 0, cols - 1)] -= 8.0 * np.float64(g[pick[i]])
    U.assert_close_stored(dX[torch.from_numpy(pick).cuda()], ref, out_fmt, 3e-6 * 8.0 * np.abs(g).max(), "xent bwd")


@pytest.mark.parametrize("rows,cols,out_fmt", [(1, 4104, "f32"), (296, 8201, "e5m2"), (297, 8201, "e5m2"), (297, 10240, "bf16"), (1000, 10247, "bf16"), (296, 16384, "f32"),
                                               (297, 16384, "f32"), (592, 8192, "f32"), (593, 8192, "f32"), (800, 4999, "e5m2"), (800, 5000, "e5m2")])
def test_softmax_xent_backward_on_both_sides_of_the_ring(rows, cols, out_fmt):
    L, synth = _mods()
    ld = (cols + 15) // 16 * 16
    x, g = synth.normal(36, cols, (rows, cols), 2.0), synth.normal(36, 1, (1, rows))[0]
    t = (np.arange(rows) * 7919 % cols).astype(np.int32)
    dX = U.empty(rows, cols, out_fmt, ld)
    L.us_softmax_xent_bwd(U.to_device(x, "bf16", ld), torch.from_numpy(t).cuda(), torch.from_numpy(g).cuda(), 8.0, dX)
    pick = np.unique(np.concatenate([np.arange(0, rows, 37), np.arange(max(0, rows - 3), rows)]))
    ref = O.softmax_xent_bwd(U.values_of(x, "bf16")[pick], t[pick], g[pick].astype(np.float64), 8.0)
    U.assert_close_stored(dX[torch.from_numpy(pick).cuda()], ref, out_fmt, 3e-6 * 8.0 * np.abs(g).max(), "xent bwd")


@pytest.mark.parametrize("rows,cols,out_fmt", [(700, 6000, "bf16"), (700, 6003, "e5m2"), (40, 12000, "f32"), (700, 3000, "bf16")])
def test_softmax_xent_backward_of_rows_that_are_not_finite(rows, cols, out_fmt):
    """A NaN, a row of -inf only and a +inf make their own row NaN, in the ring (the first three) as in registers, and no other."""
    L, synth = _mods()
    ld = (cols + 15) // 16 * 16
    x = synth.normal(37, cols, (rows, cols), 2.0)
    bad = {5: ("one", np.nan), 6: ("all", -np.inf), 7: ("one", np.inf), rows - 2: ("last", np.nan)}
    for r, (where, v) in bad.items():
        x[r, {"one": slice(cols // 3, cols // 3 + 1), "all": slice(None), "last": slice(cols - 1, cols)}[where]] = v
    x[11, ::2] = -np.inf                                                 # finite: half of the weights are zero
    t = (np.arange(rows) * 7919 % cols).astype(np.int32)
    X = torch.zeros(rows, ld, device="cuda")
    X[:, :cols] = torch.from_numpy(x).cuda()
    X = X.to(torch.bfloat16)[:, :cols]
    dX = U.empty(rows, cols, out_fmt, ld)
    L.us_softmax_xent_bwd(X, torch.from_numpy(t).cuda(), None, 8.0, dX)
    got = dX.float().cpu().numpy()
    good = np.setdiff1d(np.arange(rows), list(bad))
    assert np.isnan(got[list(bad)]).all() and np.isfinite(got[good]).all()
    pick = np.unique(np.concatenate([good[:16], good[::37], good[-3:]]))
    ref = O.softmax_xent_bwd(X.double().cpu().numpy()[pick], t[pick], np.ones(len(pick)), 8.0)
    U.assert_close_stored(dX[torch.from_numpy(pick).cuda()], ref, out_fmt, 3e-6 * 8.0, "xent bwd")


@pytest.mark.parametrize("rows,cols", [(2400, 700), (700, 3000), (700, 9001), (300, 12000), (40, 16390), (40, 30522), (12, 40000)])
@pytest.mark.parametrize("in_fmt", ["bf16", "fp16"])
def test_softmax_xent_of_rows_that_are_not_finite_in_every_form(rows, cols, in_fmt):
    """A warp per row, registers, the ring, staged rows, rows that are read again: a NaN, a +inf and a row of -inf only make the row's
    log-likelihood and gradient NaN, in the maximum of packed pairs as well; classes of -inf or of the type's lowest value (masks) have
    weight zero."""
    L, synth = _mods()
    ld = (cols + 15) // 16 * 16
    x = U.values_of(synth.normal(39, cols, (rows, cols), 2.0), in_fmt).astype(np.float32)
    bad = {3: (cols // 3, np.nan), 4: (cols - 1, np.nan), 5: (0, np.inf), 6: (slice(None), -np.inf)}
    for r, (where, v) in bad.items():
        x[r, where] = v
    x[8, 1::2] = -np.inf
    # (some classes, not all: the row's maximum times log2 e is rounded before it is subtracted, by up to 2^-8 at 65504, and overflows in BF16)
    x[9, 1::3] = -65504.0 if in_fmt == "fp16" else -3.3895314e38
    X = torch.zeros(rows, ld, device="cuda", dtype=U.TORCH_OF[in_fmt])[:, :cols]
    X.copy_(torch.from_numpy(x))
    t = (np.arange(rows) * 7919 % cols).astype(np.int32)
    t[8] = t[8] // 2 * 2
    tt, out, dX = torch.from_numpy(t).cuda(), torch.empty(rows, device="cuda"), U.empty(rows, cols, "bf16", ld)
    L.us_softmax_xent_fwd(X, tt, out)
    L.us_softmax_xent_bwd(X, tt, None, 8.0, dX)
    got, ll, good = dX.float().cpu().numpy(), out.cpu().numpy(), np.setdiff1d(np.arange(rows), list(bad))
    assert np.isnan(got[list(bad)]).all() and np.isfinite(got[good]).all()
    assert np.isnan(ll[list(bad)]).all() and np.isfinite(ll[good]).all()
    pick = np.unique(np.concatenate([good[:8], good[::53]]))
    v = X.double().cpu().numpy()[pick]
    ref = O.softmax_xent_fwd(v, t[pick])
    assert np.abs(ll[pick] - ref).max() <= 4e-6 * (1 + np.abs(ref).max())
    U.assert_close_stored(dX[torch.from_numpy(pick).cuda()], O.softmax_xent_bwd(v, t[pick], np.ones(len(pick)), 8.0), "bf16", 3e-6 * 8.0, "xent bwd")


@pytest.mark.parametrize("rows,cols,out_fmt", [(700, 3000, "bf16"), (700, 5000, "f32"), (700, 6003, "bf16"), (700, 9000, "f32"),
                                               (300, 12001, "e5m2"), (9, 20003, "f32"), (9, 40001, "bf16")])
@pytest.mark.parametrize("in_fmt", ["bf16", "fp16"])
def test_softmax_xent_backward_of_an_infinite_gradient(rows, cols, out_fmt, in_fmt):
    """beta g (onehot - p) with an infinite g (a loss that overflowed): infinite at the target and of the other sign elsewhere (saturated
    in FP8), not NaN; with a finite one a class of weight zero gets +0.  In registers, the ring, staged and read again."""
    L, synth = _mods()
    ld = (cols + 15) // 16 * 16
    x, g = synth.normal(38, cols, (rows, cols), 2.0), np.ones(rows, np.float32)
    t = (np.arange(rows) * 7919 % cols).astype(np.int32)
    t[8] = cols - 1
    g[[2, 8]], g[5] = np.inf, -np.inf
    x[3, ::2] = -np.inf
    dX = U.empty(rows, cols, out_fmt, ld)
    L.us_softmax_xent_bwd(U.to_device(x, in_fmt, ld), torch.from_numpy(t).cuda(), torch.from_numpy(g).cuda(), 8.0, dX)
    got = dX.float().cpu().numpy()
    most = 57344.0 if out_fmt == "e5m2" else np.inf
    for r in (2, 5, 8):
        want = np.full(cols, -most if g[r] > 0 else most)
        want[t[r]] *= -1
        assert np.array_equal(got[r], want)
    off = np.setdiff1d(np.arange(0, cols, 2), t[3])
    assert not got[3, off].any() and not np.signbit(got[3, off]).any()
