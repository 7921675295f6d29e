"""us_cast_fp8 against the oracle quantiser: bit-exact codes."""
import numpy as np
import pytest
import torch

from oracle import formats as F
from tests import util as U

pytestmark = pytest.mark.gpu


def _lib():
    from paper_2303_11257_b200 import lib
    return lib


def structured_fp32_patterns():
    hi = np.arange(1 << 16, dtype=np.uint32)
    lo = np.random.default_rng(4).integers(0, 1 << 16, size=256, dtype=np.uint32)
    lo[:4] = [0, 1, 0x8000, 0xFFFF]
    return (hi[:, None] << 16 | lo[None, :]).reshape(1 << 12, 1 << 12).view(np.float32)


def _assert_codes(got, want, fmt):
    nan_want = np.isnan(F.decode(want, fmt))
    nan_got = np.isnan(F.decode(got, fmt))
    assert np.array_equal(nan_want, nan_got)
    assert np.array_equal(got[~nan_want], want[~nan_want])


@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
def test_cast_structured_fp32_bit_patterns(fmt):
    L = _lib()
    x = structured_fp32_patterns()
    dst = U.empty(*x.shape, fmt)
    L.us_cast_fp8(torch.from_numpy(x).cuda(), 1.0, dst)
    _assert_codes(U.codes_of(dst), F.scaled_cast(x, 1.0, F.FORMATS[fmt]), F.FORMATS[fmt])


@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
@pytest.mark.parametrize("src", ["bf16", "fp16"])
def test_cast_all_16bit_sources(fmt, src):
    L = _lib()
    codes = np.arange(1 << 16, dtype=np.uint16).reshape(256, 256)
    t = torch.from_numpy(codes.view(np.int16)).view(U.TORCH_OF[src]).cuda()
    vals = F.decode(codes, F.FORMATS[src])
    for scale in (1.0, 0.3, 2.0 ** -7):
        dst = U.empty(256, 256, fmt)
        L.us_cast_fp8(t, scale, dst)
        with np.errstate(over="ignore", invalid="ignore"):
            want = F.scaled_cast(vals.astype(np.float32), scale, F.FORMATS[fmt])
        _assert_codes(U.codes_of(dst), want, F.FORMATS[fmt])


@pytest.mark.parametrize("fmt", ["e4m3", "e5m2"])
@pytest.mark.parametrize("shape,ld", [((1, 1), None), ((3, 5), None), ((300, 257), None), ((64, 48), 64),
                                      ((37, 100), 112), ((2048, 4096), None)])
def test_cast_shapes_scales_and_saturation(fmt, shape, ld):
    from paper_2303_11257_b200 import synth
    L = _lib()
    for sigma, scale in ((1.0, 1.0), (256.0, 1.0), (2.0 ** -8, 1.0), (1.0, 1 / 3), (1.0, 1000.0)):
        x = synth.normal(11, 0, shape, sigma)
        src = U.to_device(x, "f32", ld)
        dst = U.empty(shape[0], shape[1], fmt, ld)
        L.us_cast_fp8(src, scale, dst)
        want = F.scaled_cast(x, scale, F.FORMATS[fmt])
        assert np.array_equal(U.codes_of(dst), want)
        if ld:   # padding untouched
            full = dst.as_strided((shape[0], ld), (ld, 1)).view(torch.uint8).cpu().numpy()
            assert not full[:, shape[1]:].any()


@pytest.mark.parametrize("shape,ld", [((2500, 2007), 2016), ((700, 16001), 16016), ((1, 4099), None)])
@pytest.mark.parametrize("src", ["f32", "bf16"])
def test_cast_of_padded_rows_with_several_chunks_per_thread(shape, ld, src):
    """More chunks than resident threads, row ends inside a chunk, and nothing written behind a row's end."""
    from paper_2303_11257_b200 import synth
    L = _lib()
    x = synth.normal(12, 0, shape)
    dst = U.empty(*shape, "e4m3", ld)
    L.us_cast_fp8(U.to_device(x, src, ld), 0.75, dst)
    assert np.array_equal(U.codes_of(dst), F.scaled_cast(U.values_of(x, src).astype(np.float32), 0.75, F.E4M3))
    if ld:
        assert not dst.as_strided((shape[0], ld), (ld, 1)).view(torch.uint8)[:, shape[1]:].any()


@pytest.mark.parametrize("src", ["f32", "bf16", "fp16"])
@pytest.mark.parametrize("shape,ld", [((70, 32), 48), ((70, 33), 48), ((70, 100), 112), ((70, 101), 112), ((1, 100), 112), ((700, 101), 101), ((3, 20), 32)])
def test_cast_on_both_sides_of_the_choice_of_kernel(shape, ld, src):
    from paper_2303_11257_b200 import synth
    L = _lib()
    x = synth.normal(13, 0, shape)
    dst = U.empty(*shape, "e5m2", ld)
    L.us_cast_fp8(U.to_device(x, src, ld), 1.5, dst)
    assert np.array_equal(U.codes_of(dst), F.scaled_cast(U.values_of(x, src).astype(np.float32), 1.5, F.E5M2))


def test_cast_empty_and_errors():
    L = _lib()
    src = torch.zeros((0, 8), device="cuda")
    dst = torch.zeros((0, 8), dtype=torch.uint8, device="cuda").view(torch.float8_e4m3fn)
    L.us_cast_fp8(src, 1.0, dst)
    with pytest.raises(L.UnitScaleError) as e:
        L.us_cast_fp8(torch.zeros((4, 8), device="cuda"), 1.0, torch.zeros((4, 8), device="cuda", dtype=torch.bfloat16))
    assert e.value.status == 2
    with pytest.raises(L.UnitScaleError) as e:
        L.us_cast_fp8(torch.zeros((4, 8), device="cuda"), 1.0, U.empty(4, 9, "e4m3"))
    assert e.value.status == 1


def test_cast_multi_matches_oracle_and_single_casts():
    """Mixed source types, formats, scales and ragged sizes in one launch: codes equal the oracle's and
    those of separate us_cast_fp8 calls; neighbours of each destination stay untouched."""
    from paper_2303_11257_b200 import synth
    L = _lib()
    specs = [((64, 48), "f32", "e4m3", 1.0), ((1, 1), "f32", "e5m2", 0.5), ((300, 257), "bf16", "e5m2", 3.0),
             ((37, 19), "fp16", "e4m3", 2.0 ** -3), ((0, 8), "f32", "e4m3", 1.0), ((1024, 1024), "f32", "e4m3", 1 / 3),
             ((5, 16), "bf16", "e4m3", 1000.0), ((2, 7), "f32", "e5m2", 1.0)]
    srcs, dsts, wants, singles, scales = [], [], [], [], []
    for i, (shape, st, fmt, scale) in enumerate(specs):
        x = synth.normal(21 + i, 0, shape, 4.0)
        xs = F.quantise(x, F.FORMATS[st]).astype(np.float32) if st != "f32" else x
        srcs.append(U.to_device(xs, st) if x.size else torch.zeros(shape, device="cuda"))
        dsts.append(U.empty(shape[0], shape[1], fmt))
        singles.append(U.empty(shape[0], shape[1], fmt))
        wants.append(F.scaled_cast(xs, scale, F.FORMATS[fmt]))
        scales.append(scale)
    L.us_cast_fp8_multi(srcs, scales, dsts)
    for src, scale, one in zip(srcs, scales, singles):
        L.us_cast_fp8(src, scale, one)
    for dst, one, want in zip(dsts, singles, wants):
        assert np.array_equal(U.codes_of(dst), want)
        assert np.array_equal(U.codes_of(dst), U.codes_of(one))


def test_cast_multi_errors_launch_nothing():
    L = _lib()
    a, b = torch.ones((4, 16), device="cuda"), torch.ones((4, 16), device="cuda")
    da, db = U.empty(4, 16, "e4m3"), U.empty(4, 16, "e4m3")
    da.view(torch.uint8).zero_()
    padded = U.empty(4, 16, "e4m3", 32)
    with pytest.raises(L.UnitScaleError) as e:                       # row padding: not for the fused launch
        L.us_cast_fp8_multi([a, b], [1.0, 1.0], [da, padded])
    assert e.value.status == 2
    with pytest.raises(L.UnitScaleError) as e:                       # shape mismatch
        L.us_cast_fp8_multi([a, b], [1.0, 1.0], [da, U.empty(4, 8, "e4m3")])
    assert e.value.status == 1
    with pytest.raises(L.UnitScaleError) as e:                       # more tensors than one launch takes
        L.us_cast_fp8_multi([a] * 9, [1.0] * 9, [da] * 9)
    assert e.value.status == 1
    with pytest.raises(L.UnitScaleError) as e:                       # misaligned start
        L.us_cast_fp8_multi([a.view(-1)[1:33].view(2, 16)], [1.0], [U.empty(2, 16, "e4m3")])
    assert e.value.status == 3
    torch.cuda.synchronize()
    assert not da.view(torch.uint8).any()                            # the valid first tensor was not written either


@pytest.mark.parametrize("src_fmt", ["f32", "bf16"])
def test_cast_multi_into_padded_rows(src_fmt):
    """Destinations with padded rows beside dense ones, one row, more chunks than a grid takes at once: the codes of single casts, and
    nothing written between the rows; what the other forms refuse stays refused."""
    from paper_2303_11257_b200 import lib as L, synth
    shapes = [(5, 16, 32, "e4m3"), (1, 144, 256, "e5m2"), (3000, 528, 640, "e4m3"), (64, 96, 96, "bf16"), (33, 272, 384, "fp16"), (70, 100, 100, "e4m3")]
    srcs = [U.to_device(synth.normal(21, i, (r, c)), src_fmt) for i, (r, c, _, _) in enumerate(shapes)]
    outs = [[U.empty(r, c, f, ld) for r, c, ld, f in shapes] for _ in range(2)]
    L.us_cast_multi_pitched(srcs, [1.0, 0.5, 1.0, 1.0, 1.0, 2.0], outs[0])
    for s, o, k, (r, c, ld, f) in zip(srcs, outs[1], [1.0, 0.5, 1.0, 1.0, 1.0, 2.0], shapes):
        L.us_cast_fp8(s, k, o) if f[0] == "e" else L.us_residual_add(s, s, 0.0, o)
    for a, b, (r, c, ld, f) in zip(*outs, shapes):
        assert np.array_equal(U.codes_of(a), U.codes_of(b))
        assert not a.as_strided((r, ld), (ld, 1))[:, c:].contiguous().view(torch.uint8).any()

    def status(s, d):
        with pytest.raises(L.UnitScaleError) as e:
            L.us_cast_multi_pitched([s], [1.0], [d])
        return e.value.status

    padded = U.to_device(synth.normal(21, 9, (8, 32)), src_fmt, 48)
    assert status(padded, U.empty(8, 32, "e4m3", 48)) == L.US_ERR_UNSUPPORTED                # padded sources
    assert status(srcs[5], U.empty(70, 100, "e4m3", 112)) == L.US_ERR_UNSUPPORTED            # rows that end inside a chunk
    assert status(srcs[0], U.empty(5, 16, "e4m3", 24)) == L.US_ERR_ALIGNMENT                 # row starts
    with pytest.raises(L.UnitScaleError):
        L.us_cast_multi([srcs[0]], [1.0], [outs[0][0]])
