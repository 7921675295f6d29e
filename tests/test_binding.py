"""The Python binding's argument conversion and prepared passes, without a GPU: every call here is refused by the library's host
checks, or by the binding itself, before anything is launched."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2303_11257_b200 import _binding
from paper_2303_11257_b200 import lib as L

cast = _binding.calls["us_cast_fp8"]
F32, F8 = torch.zeros(4, 16), torch.zeros(4, 16, dtype=torch.float8_e4m3fn)


@pytest.mark.parametrize("bad,error", [(5, TypeError), (np.zeros((4, 16), np.float32), TypeError), ([F32], TypeError), (torch.zeros(16), ValueError),
                                       (torch.zeros(16, 4).t(), ValueError), (torch.zeros(4, 16, dtype=torch.int64), KeyError)])
def test_what_is_no_matrix_is_refused_by_the_binding(bad, error):
    with pytest.raises(error):
        cast(bad, 1.0, F8, 0)


def test_argument_counts_and_numbers_are_checked():
    for args in ((F32, 1.0, F8), (F32, 1.0, F8, 0, 0), (F32, "1", F8, 0), (F32, 1.0, F8, "0")):
        with pytest.raises(TypeError):
            cast(*args)
    with pytest.raises(KeyError):
        _binding.prepare("us_nothing", ())


@pytest.mark.parametrize("t", [F32, F32[:, :5], F32[:1, :5], torch.zeros(1, 1), F32.to(torch.bfloat16)[1:3]])
def test_a_tensor_is_described_as_by_the_python_side(t):
    """A slot of a program gets what describe() says (the call itself is refused: its output has another shape)."""
    m, out = L.us_mat(), L.mat(torch.zeros(7, 3, dtype=torch.float8_e4m3fn))
    prog = _binding.program([(0, _binding.prepare("us_cast_fp8", (m, 1.0, out)))], [(0, m)])
    assert _binding.run(prog, 0, (t,), 0, 0, 0, 0) == L.US_ERR_INVALID_ARG
    assert (m.ptr, m.dtype, m.rows, m.cols, m.ld) == L.describe(t)


def test_a_pass_stops_at_a_refused_call_and_goes_on_behind_it():
    bad, good = L.mat(F32), L.mat(torch.zeros(4, 16, dtype=torch.bfloat16))
    empty = L.us_mat(None, L.US_F32, 0, 16, 16)
    nothing = _binding.prepare("us_cast_fp8", (empty, 1.0, L.us_mat(None, L.US_E4M3, 0, 16, 16)))      # no rows: succeeds, launches nothing
    refused = _binding.prepare("us_cast_fp8", (bad, 1.0, good))                                        # no 8-bit output
    prog = _binding.program([(0, nothing), (0, refused), (2, None), (0, nothing), (1, refused)], [])
    assert _binding.run(prog, 0, (), 0, 0, 0, 0) == 1 << 8 | L.US_ERR_UNSUPPORTED
    assert _binding.run(prog, 2, (), 0, 0, 0, 0) == 4 << 8 | L.US_ERR_UNSUPPORTED
    assert _binding.run(prog, 5, (), 0, 0, 0, 0) == -1


def test_unchanged_compares_objects_and_addresses():
    own = (F32, F8)
    at = tuple(t.data_ptr() for t in own)
    assert _binding.unchanged(own, own, at)
    assert not _binding.unchanged((F32, F8.clone()), own, at) and not _binding.unchanged(own, own, (at[0], at[1] + 16)) and not _binding.unchanged(own[:1], own, at)


def test_fp8_copies_are_validated_before_any_launch():
    """Statuses of the entry points that leave an FP8 copy (1 invalid argument, 2 unsupported, 3 alignment); fake device addresses."""
    M = lambda addr, dt, r, c, ld=None: L.us_mat(addr, dt, r, c, ld or c)
    X, W, Y = M(0x10000, L.US_E4M3, 64, 32), M(0x20000, L.US_E4M3, 32, 48), M(0x30000, L.US_BF16, 64, 48)
    ep, no = L.us_epilogue(), L.us_epilogue()
    ep.skip, ep.skip_coef, ep.out_coef = M(0x40000, L.US_BF16, 64, 48), 0.5, 0.5
    fwd = lambda e, y, q: _binding.calls["us_linear_fwd_cast"](X, W, 1.0, e, y, q, 0x60000, 256, 0)
    good = M(0x50000, L.US_E4M3, 64, 48)
    assert fwd(ep, Y, None) == 1 and fwd(ep, Y, M(0x50000, L.US_E4M3, 64, 32)) == 1
    assert fwd(no, Y, good) == 2 and fwd(None, Y, good) == 2                     # no skip tensor
    assert fwd(ep, Y, M(0x50000, L.US_BF16, 64, 48)) == 2                        # the copy is FP8 ...
    assert fwd(ep, M(0x30000, L.US_E5M2, 64, 48), good) == 2                     # ... of something that is not
    assert fwd(ep, Y, M(0x50008, L.US_E4M3, 64, 48)) == 3
    v = M(0x70000, L.US_F32, 1, 48)
    norm = lambda y, q: _binding.calls["us_layer_norm_fwd_cast"](M(0x10000, L.US_BF16, 64, 48), v, v, 1e-5, y, q, 0)
    assert norm(Y, None) == 1 and norm(Y, M(0x50000, L.US_E4M3, 64, 32)) == 1 and norm(Y, M(0x50000, L.US_BF16, 64, 48)) == 2
    assert norm(M(0x30000, L.US_E5M2, 64, 48), good) == 2


ROWS = torch.zeros(4, 64, dtype=torch.bfloat16)
WS = torch.zeros(256, dtype=torch.uint8)
ONE, TWO = L.us_mat(0x10000, L.US_F32, 4, 16, 16), (L.us_mat * 2)()
WRONG = [L.us_mat(), L.us_epilogue(), L.us_batch(), L.us_attention_batch(), L.us_attention_bwd_batch(), L.us_attention_bwd_all_batch(), C.c_float(1.0),
         C.c_void_p(0x10000), C.pointer(L.us_mat()), C.byref(L.us_mat()), (C.c_uint8 * 4096)(), (L.us_epilogue * 2)(), b"x" * 4096, np.zeros(4096, np.uint8)]


@pytest.mark.parametrize("call,own", [
    (lambda x: L.us_attention_fwd(ROWS, ROWS, ROWS, 1.0, 1.0, 1.0, ROWS, None, x, WS, 0), L.us_attention_batch),
    (lambda x: L.us_attention_bwd(ROWS, ROWS, ROWS, ROWS, 1.0, 1.0, 1.0, 1.0, ROWS, ROWS, x, WS, 0), L.us_attention_bwd_batch),
    (lambda x: L.us_attention_bwd_all(ROWS, ROWS, ROWS, ROWS, ROWS, *[1.0] * 6, ROWS, ROWS, ROWS, ROWS, x, WS, 0), L.us_attention_bwd_all_batch),
    (lambda x: L.us_linear_fwd_batched(ROWS, ROWS, 1.0, ROWS, x, WS, 0), L.us_batch),
    (lambda x: L.us_linear_fwd(F32, F32, 1.0, F32, WS, x, 0), L.us_epilogue),
    (lambda x: cast(x, 1.0, F8, 0), L.us_mat),
    (lambda x: L.us_linear_fwd(F32, F32, 1.0, F32, x, None, 0), None),                      # the workspace
    (lambda x: _binding.program([], [(0, x)]), L.us_mat)])
def test_a_structure_of_another_kind_is_refused(call, own):
    for x in WRONG:
        if own is not None and type(x) in (own, own * 2):
            continue
        with pytest.raises((TypeError, AttributeError, KeyError)):
            call(x)


def test_arrays_hold_as_many_elements_as_the_count():
    calls, factors = (L.us_linear_call * 2)(), (C.c_float * 2)(1.0, 1.0)
    for args in [("us_linear_group", 3, calls, WS, WS), ("us_linear_group_any", 2, calls[0], WS, WS), ("us_linear_group_cast", 2, calls, ONE, WS, WS),
                 ("us_cast_fp8_multi", 3, (L.us_mat * 3)(), factors, (L.us_mat * 3)()), ("us_cast_multi", 2, TWO, factors, ONE), ("us_weighted_add", 2, ONE, factors, 1.0, ONE)]:
        with pytest.raises(ValueError):
            _binding.calls[args[0]](*args[1:], 0)
        with pytest.raises(ValueError):
            _binding.prepare(args[0], tuple(a if a is not WS else 256 for a in args[1:]))
    for factor in (0x10000, F32):                                                           # numbers on the host, not an address
        with pytest.raises(TypeError):
            _binding.calls["us_weighted_add"](2, TWO, factor, 1.0, ONE, 0)
    assert _binding.calls["us_weighted_add"](2, TWO, factors, 1.0, ONE, 0) == L.US_ERR_INVALID_ARG
    assert _binding.calls["us_linear_group"](0, calls, WS, WS, 0) == L.US_ERR_INVALID_ARG


@pytest.mark.parametrize("ws", [0x10000, 4096, None, np.zeros(256, np.uint8)])
def test_a_workspace_is_a_tensor(ws):
    """An address alone says nothing about the size; it is not taken for one."""
    with pytest.raises(TypeError):
        L.us_linear_fwd(F32, F32, 1.0, F32, ws, None, 0)
    with pytest.raises(TypeError):
        L.us_linear_group([L.us_linear_call()], ws, 0)
